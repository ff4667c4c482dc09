// The whole decode step of a shard as one persistent, cooperative kernel.
//
// One CTA per SM, whose warps stream their weights into rings of their own
// (gemv_core.cuh).  The step runs as a sequence of phases separated by grid-wide
// barriers ('|'):
//   prologue (every CTA: its share of the beam-table gather, the new
//   entries' slots and the residual) ~ for each layer: RMSNorm + q|k|v
//   projection -> attention (chunk partials and merges, with RoPE and the K/V
//   append) | o projection (+residual) | RMSNorm + gate|up projection
//   (+SwiGLU) | down projection (+residual) | ... ; then hidden_out.
// '~' is a split barrier: CTAs arrive after their prologue share and wait only
// before the first attention, so the first norm and q|k|v projection overlap
// the prologue.  '->' is dataflow: q|k|v contributors count finished units
// per kv head (release) and an attention unit waits (acquire, bounded) only
// for its kv head's count.
//
// The residual stream and the projections' sums are 64-bit fixed point
// (kernels.h): contributors add with integer atomics and nobody waits for a
// merge; results do not depend on the order of arrival.
// Each RMSNorm runs at the start of the projection that consumes it: one row by
// every CTA for itself, several by one CTA each.
//
// Every cross-CTA wait is bounded: a wait that runs out sets a status bit and
// proceeds (the step's results are then reported invalid) instead of hanging.
#include <type_traits>

#include <algorithm>

#include "gemv_core.cuh"

namespace shard {
namespace {

constexpr int kWarps = kCtaWarps;
constexpr int kThreads = kWarps * 32;

// Dynamic shared memory: weight rings, their barriers, the op table (4L
// entries), gate|up partial sums (when they fit), and the area: an attention
// unit's (AttnSmem), which between attentions holds the normalised rows when
// they fit.  The host sizes the area for the step's token count.
constexpr size_t kAttnArea = 51 * 1024;  // at least: AttnSmem at head_dim 128, checked in the kernel

template <int GPU>
struct StepSmem {
  static constexpr int kSlots = Geom<GPU>::kStepSlots;
  static constexpr size_t kRing = (size_t)kWarps * kSlots * Geom<GPU>::kUnitBytes;
  static constexpr size_t kBars = (size_t)kWarps * kSlots * sizeof(uint64_t);
  static constexpr size_t kOps = kRing + kBars;
  // gate|up partial sums of the shared-memory reduction (swiglu_cta_write) for M tokens
  __host__ __device__ static size_t part(int M) { return (size_t)kWarps * M * kRowsPerBlock * sizeof(float); }
  // offset of the area
  __host__ __device__ static size_t area(int n_layers, bool with_part, int M) {
    return (kOps + (size_t)4 * n_layers * sizeof(OpDesc) + (with_part ? part(M) : 0) + 127) / 128 * 128;
  }
};

// Row stride (halves) of the normalised rows in shared memory: padded so that
// the two token rows a fragment load touches in one phase fall on different
// banks.
__host__ __device__ constexpr int xn_stride(int H) { return H + 32; }
// Bytes of M such rows, and of the one residual row staged behind them when M = 1.
__host__ __device__ constexpr size_t xn_bytes(int H, int M) { return ((size_t)M * xn_stride(H) * 2 + 127) / 128 * 128; }
__host__ __device__ constexpr size_t xn_stage_bytes(int H, int M) { return M == 1 ? (size_t)H * 8 : 0; }

// The same value, which the compiler may not trace to where it came from.  The
// phases of the layer loop start from such values: it would otherwise compute
// their address parts before the loop and hold them in registers (or spill
// them) through all the other phases.
__device__ __forceinline__ int opaque(int v) {
  asm volatile("" : "+r"(v));
  return v;
}

// Barrier among the warps of a CTA.
__device__ __forceinline__ void cbar() { named_bar_sync(1, kThreads); }

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ float2 h2f2(uint32_t u) {
  __half2 h;
  memcpy(&h, &u, sizeof(h));
  return __half22float2(h);
}

// two floats rounded to fp16 (to nearest even), lo in the low half
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
  return (uint32_t)f2h(lo) | ((uint32_t)f2h(hi) << 16);
}

__device__ __forceinline__ void red_release_add(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Grid-wide barrier on a monotonically increasing counter, in two halves so
// that work may sit between arriving and waiting.  `target` is this CTA's
// running count of expected arrivals.  The caller has
// synchronised the CTA (cbar) before grid_arrive.  Lives in shared
// memory (only thread 0 uses it), so that it takes no registers of the phases.
struct GridBarrier {
  unsigned long long* ctr;
  unsigned long long target;
  int* status;
  unsigned long long* clock;
  int n_arrive, n_wait;
  int skip_arrival;  // test knob: CTA 1 leaves out this arrival (-1: none)
  uint32_t limit;

  __device__ __forceinline__ void arrive() {
    if (threadIdx.x == 0) {
      if (!(blockIdx.x == 1 && n_arrive == skip_arrival)) red_release_add(ctr, 1ULL);
      ++n_arrive;
    }
  }
  __device__ __forceinline__ void wait() {
    if (threadIdx.x == 0) {
      target += gridDim.x;
      // bounded: after `limit` polls, or once any CTA has given up, stop waiting
      uint32_t it = 0;
      while (ld_acquire_u64(ctr) < target) {
        if (++it > limit) {
          atomicOr(status, ST_WAIT_TIMEOUT);
          break;
        }
        if ((it & 1023) == 0 && (*reinterpret_cast<volatile int*>(status) & ST_WAIT_TIMEOUT)) break;
        __nanosleep(16);
      }
      if (blockIdx.x == 0) clock[++n_wait] = globaltimer();
    }
    cbar();
  }
  __device__ __forceinline__ void sync() {
    cbar();
    arrive();
    wait();
  }
};

__device__ __forceinline__ bool wait_count(const int* p, int target, int* status, uint32_t limit) {
  uint32_t it = 0;
  while (ld_acquire_s32(p) < target) {
    if (++it > limit) {
      atomicOr(status, ST_WAIT_TIMEOUT);
      return false;
    }
    if ((it & 1023) == 0 && (*reinterpret_cast<volatile int*>(status) & ST_WAIT_TIMEOUT)) return false;
    __nanosleep(20);
  }
  return true;
}

// ---------------------------------------------------------------------------
// Prologue, part 1 (every CTA, all threads): the step's bookkeeping from its
// arguments -- Section 4's beam_idx gather (row b continues row beam_idx[b]'s
// entries; K/V stay where they are), the new entries' slots -- and the
// device-side argument checks.  Every CTA derives the same values.
// ---------------------------------------------------------------------------
// `plan` runs on warp 2 once the lengths are known, behind the other checks' loads.
template <class Plan>
__device__ __noinline__ void prologue_params(const PrologueArgs& a, StepParams* sp, const uint16_t** rowp,
                                             const Plan& plan) {
  __shared__ int s_err;
  const int tid = threadIdx.x;
  if (tid == 0) {
    // a step rejected earlier freezes the state until the host resets it
    s_err = __ldcg(a.status) != 0 ? ST_STICKY : 0;
    int t = 0;
    for (int b = 0; b < a.B; ++b) {
      sp->req_tok0[b] = t;
      for (int i = 0; i < a.n_new[b]; ++i, ++t) {
        sp->tok_req[t] = b;
        sp->tok_idx[t] = i;
      }
    }
    sp->req_tok0[a.B] = t;
    sp->M = a.M;
    sp->B = a.B;
  }
  __syncthreads();
  if (tid < a.B) {
    int src = a.beam_idx ? __ldcg(a.beam_idx + tid) : tid;
    if (src < 0 || src >= a.B) {
      atomicOr(&s_err, ST_BEAM_IDX);
      src = tid;
    }
    sp->req_src[tid] = src;
    const int P = __ldcg(a.lens + src);
    const int L = P + a.n_new[tid];
    if (L > a.cap || a.cursor[tid] + a.n_new[tid] > a.cap) atomicOr(&s_err, ST_CAPACITY);
    if (L > a.mask_stride) atomicOr(&s_err, ST_MASK_STRIDE);
    sp->req_P[tid] = P;
    sp->req_len[tid] = L;
  }
  __syncthreads();
  if (tid >> 5 == 2) plan(tid & 31);
  if (tid < a.M) {
    const int m = tid, b = sp->tok_req[m], i = sp->tok_idx[m], j = sp->req_P[b] + i;
    // a token must see its own entry (packed: in its own mask row, Section 8.6)
    const size_t mrow = a.packed ? (size_t)m : (size_t)b;
    if (j < a.mask_stride && __ldcg(a.mask + mrow * a.mask_stride + j) == 0) atomicOr(&s_err, ST_MASK_NEW);
    const int pos = __ldcg(a.position_ids + m);
    if (pos < 0 || pos >= a.max_position) atomicOr(&s_err, ST_POSITION);
    sp->tok_pos[m] = pos;
    sp->tok_slot[m] = b * a.cap + a.cursor[b] + i;
    if (a.token_ids) {
      const int tok = __ldcg(a.token_ids + m);
      if (tok < 0 || tok >= a.vocab) atomicOr(&s_err, ST_TOKEN);
      rowp[m] = a.embedding + (size_t)(tok < 0 || tok >= a.vocab ? 0 : tok) * a.H;
    } else {
      rowp[m] = a.hidden_in + (size_t)m * a.H;
    }
  }
  __syncthreads();
  if (tid == 0) sp->abort_step = s_err;
  __syncthreads();
}

// Prologue, part 2 (the threads of every CTA, a share each): the beam
// table's gather and appends, and the residual stream X = the fp16 inputs in
// fixed point (exact).
__device__ __noinline__ void prologue_work(const PrologueArgs& a, const StepParams* sp, const uint16_t* const* rowp,
                                           long long* X) {
  const int tid = threadIdx.x;
  const int gt = blockIdx.x * kThreads + tid, gs = gridDim.x * kThreads;
  if (a.beam_idx) {
    for (int b = 0; b < a.B; ++b) {
      const int* src = a.bt_src + (size_t)sp->req_src[b] * a.cap;
      int* dst = a.bt_dst + (size_t)b * a.cap;
      for (int j = gt; j < sp->req_P[b]; j += gs) dst[j] = __ldcg(src + j);
    }
  }
  if (blockIdx.x == 0 && tid < a.M) {
    const int b = sp->tok_req[tid], i = sp->tok_idx[tid];
    a.bt_dst[(size_t)b * a.cap + sp->req_P[b] + i] = sp->tok_slot[tid];
  }
  const int H4 = a.H / 4;
  for (int e = gt; e < a.M * H4; e += gs) {
    const int m = e / H4, k = 4 * (e % H4);
    const uint2 v = *reinterpret_cast<const uint2*>(rowp[m] + k);
    const float2 f01 = h2f2(v.x), f23 = h2f2(v.y);
    longlong2* dst = reinterpret_cast<longlong2*>(X + (size_t)m * a.H + k);
    dst[0] = make_longlong2(to_fixed(f01.x), to_fixed(f01.y));
    dst[1] = make_longlong2(to_fixed(f23.x), to_fixed(f23.y));
  }
}

// ---------------------------------------------------------------------------
// RMSNorm at the start of the projection that consumes it:
// r[m] = 1 / sqrt(mean(x[m]^2) + eps), act = fp16(x * r * w).  x is the
// residual stream (fixed point) or, before the first layer, the step's fp16
// input rows (the same values).  H is a multiple of 4.
//
// A single row that fits is normalised by every CTA for itself
// (rmsnorm_staged): one memory round trip and no hand-over.  Otherwise row m
// is normalised by CTA m alone, and the others wait for the count of finished
// rows and read the fp16 result: every CTA reading all M rows of 64-bit sums
// (H * 8 bytes each, 39 MB over the chip for 8 rows of 4096) costs more than
// that hand-over (8B width, norm + gate|up: 5 rows 26.6 -> 18.4 us, 8 rows
// 40 -> 19, 16 rows 80 -> 30, together with the gate|up reduction).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float4 norm_load(bool from_x, const long long* X, const uint16_t* const* rowp, int H, int m,
                                            int k) {
  if (from_x) {
    const longlong2* p = reinterpret_cast<const longlong2*>(X + (size_t)m * H + k);
    const longlong2 a = __ldcg(p), b = __ldcg(p + 1);
    return make_float4(fixed_to_f32(a.x), fixed_to_f32(a.y), fixed_to_f32(b.x), fixed_to_f32(b.y));
  } else {
    const uint2 v = *reinterpret_cast<const uint2*>(rowp[m] + k);
    const float2 f01 = h2f2(v.x), f23 = h2f2(v.y);
    return make_float4(f01.x, f01.y, f23.x, f23.y);
  }
}

// Row m to `out` (fp16), counted in *done (release) if given.  kP pieces
// (float4) per thread stay in registers between the sum of squares and the
// scaling; the rest of a longer row is read twice.
__device__ __forceinline__ void rmsnorm_row(bool from_x, const long long* X, const uint16_t* const* rowp, int H, int m,
                                            const uint16_t* w, float eps, uint16_t* out, int* done) {
  constexpr int kP = 6;
  __shared__ float s_part[kWarps];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H4 = H / 4;
  uint2 wv[kP];
  float4 v[kP];
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kThreads;
    wv[i] = c < H4 ? *reinterpret_cast<const uint2*>(w + 4 * c) : make_uint2(0, 0);
    v[i] = c < H4 ? norm_load(from_x, X, rowp, H, m, 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < kP; ++i) t += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  for (int c = tid + kP * kThreads; c < H4; c += kThreads) {
    const float4 u = norm_load(from_x, X, rowp, H, m, 4 * c);
    t += u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) s_part[warp] = t;
  cbar();
  float u = 0.f;
  for (int w8 = 0; w8 < kWarps; ++w8) u += s_part[w8];
  const float r = rsqrtf(u / H + eps);
  auto emit = [&](int c, float4 x, uint2 wq) {
    const float2 w01 = h2f2(wq.x), w23 = h2f2(wq.y);
    uint2 o;
    o.x = pack_h2(x.x * r * w01.x, x.y * r * w01.y);
    o.y = pack_h2(x.z * r * w23.x, x.w * r * w23.y);
    *reinterpret_cast<uint2*>(out + 4 * c) = o;
  };
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kThreads;
    if (c < H4) emit(c, v[i], wv[i]);
  }
  for (int c = tid + kP * kThreads; c < H4; c += kThreads)
    emit(c, norm_load(from_x, X, rowp, H, m, 4 * c), *reinterpret_cast<const uint2*>(w + 4 * c));
  cbar();
  if (done && tid == 0) red_release_add_s32(done, 1);
}

// One row from the residual stream (M = 1, H <= 24 * kThreads) through
// shared memory: the row's H fixed-point values arrive with bulk copies
// (`stage`, 16-byte aligned, H * 8 bytes; completion on `bar`, whose phase
// the caller tracks), so the read runs at copy-engine bandwidth instead of
// being bounded by each thread's loads in flight; both passes then read
// shared memory.  The values and the arithmetic are those of rmsnorm_row.
__device__ __forceinline__ void rmsnorm_staged(const long long* X, int H, const uint16_t* w, float eps, uint16_t* out,
                                               long long* stage, uint64_t* bar, uint32_t& phase, int* status) {
  constexpr int kP = 6;
  constexpr uint32_t kPiece = 8192;  // bytes per bulk copy
  __shared__ float s_part[kWarps];
  __shared__ float s_r;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H4 = H / 4;
  if (tid == 0) {
    // X was written through the generic proxy (made visible by the grid
    // barrier); the area was last used by generic accesses of this CTA
    asm volatile("fence.proxy.async;" ::: "memory");
    const uint32_t bytes = (uint32_t)H * 8u;
    mbar_arrive_expect_tx(bar, bytes);
    for (uint32_t off = 0; off < bytes; off += kPiece)
      bulk_g2s(reinterpret_cast<uint8_t*>(stage) + off, reinterpret_cast<const uint8_t*>(X) + off,
               bytes - off < kPiece ? bytes - off : kPiece, bar);
  }
  uint2 wv[kP];
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kThreads;
    wv[i] = c < H4 ? *reinterpret_cast<const uint2*>(w + 4 * c) : make_uint2(0, 0);
  }
  if (!mbar_wait(bar, phase) && tid == 0) atomicOr(status, ST_WAIT_TIMEOUT);
  phase ^= 1u;
  float4 v[kP];
  float t = 0.f;
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kThreads;
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < H4) {
      const longlong2 a = reinterpret_cast<const longlong2*>(stage)[2 * c];
      const longlong2 b = reinterpret_cast<const longlong2*>(stage)[2 * c + 1];
      v[i] = make_float4(fixed_to_f32(a.x), fixed_to_f32(a.y), fixed_to_f32(b.x), fixed_to_f32(b.y));
    }
    t += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) s_part[warp] = t;
  cbar();
  if (tid == 0) {
    float u = 0.f;
    for (int w8 = 0; w8 < kWarps; ++w8) u += s_part[w8];
    s_r = rsqrtf(u / H + eps);
  }
  cbar();
  const float r = s_r;
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kThreads;
    if (c < H4) {
      const float2 w01 = h2f2(wv[i].x), w23 = h2f2(wv[i].y);
      uint2 o;
      o.x = pack_h2(v[i].x * r * w01.x, v[i].y * r * w01.y);
      o.y = pack_h2(v[i].z * r * w23.x, v[i].w * r * w23.y);
      *reinterpret_cast<uint2*>(out + 4 * c) = o;
    }
  }
  cbar();
}

// ---------------------------------------------------------------------------
// Attention.  Chunk = (request b, kv head hk, cs entries): cs is the smallest
// multiple of 16, from kAttnChunkMin up, that gives no more chunks than CTAs for
// that row alone (the whole row when it has more kv heads than that).  A chunk's
// result, and the order in which a row's chunks meet, depend on the row's length
// and queries only, so a row has the same bits alone and in any batch.  A CTA
// takes a unit, a run of chunks of one (request, kv head): one each while all
// rows' chunks find a CTA, longer runs (the same share of entries for every CTA)
// when they do not; when there are more (request, kv head) pairs than CTAs, a unit
// is a whole row and CTAs take several.
//
// The bound is the K/V stream (32 KB per 64 entries of a head at d = 128, each
// byte read once) and, for short caches, the chain of dependent L2 round
// trips.  Both products run on mma.sync straight from registers:
//   - a warp takes blocks of 16 entries; a lane's K fragment is 16 consecutive
//     bytes of an entry's row (the head dimension is summed in that order on
//     both sides), its V fragment the same 16 bytes of four entries,
//     interleaved by byte permutes, so K and V go from global memory to the
//     tensor cores without passing through shared memory, and every warp
//     keeps its next block's rows in flight while it works on the last;
//   - queries go in tiles of 8: a tile's 16 MMA rows are the 8 queries' fp16
//     values and what that rounding left out (after scaling each query by a
//     power of two to a largest value in [1, 2)), 22 to 23 bits of the row's
//     largest value at one MMA per tile; probabilities (times 2^12) are split
//     the same way for the value sum.  Sums are fp32, the softmax is online per
//     warp.  Against 64 bits the outputs before rounding are about half as far off
//     as with fp32 queries and probabilities in chains of FMAs (2.1e-3..9.3e-3 of
//     the fp16 outputs rounded the other way, now 1.2e-3..3.8e-3; 30..4000 entries,
//     1..16 tokens, scores of deviation 1 and 6).
// A warp holds one query tile; kWarps / tiles warps side by side take different
// blocks (a tile's blocks meet the other tiles' reads of them in L1), and the
// CTA adds a chunk's pieces in shared memory in a fixed order (in a run of chunks a
// warp works through a tile of a chunk alone, attn_run).  Two tiles per warp
// would halve the L1 reads, but their accumulators and the rows in flight do
// not fit 168 registers.  Chunks of one (request, kv head) meet in `part`: the CTA
// that finishes the last one merges when that is little to read, else every unit's
// CTA waits for the others and merges its share of the queries.  Steps of one
// request and of several are kernels of their own (kMany): with both in one, its
// registers and code made every step 2 to 4 % slower.
//
// First layer's attention phase, against the CUDA-core version before it (a warp
// per query over 64-entry tiles in shared memory, a CTA's tiles one after
// another): 70B width, 4096 entries, 1 token 38 -> 16 us, 5 tokens 113 -> 29;
// 8B width, 8 requests of 640..1642 entries 69 -> 23, 16 packed tokens over
// 1024 entries 73 -> 26, 5 tokens over 512 entries 20 -> 13, 1 token over 72..327
// entries 9 -> 9 (there it is the latency of the waits).
// ---------------------------------------------------------------------------
// A partial is (max, sum of exp, 2 unused, unnormalised output[d]): the
// output starts 16-byte aligned.
__host__ __device__ constexpr int part_stride(int d) { return d + 4; }

constexpr int kAttnQ = 64;        // queries per pass over a chunk's entries
constexpr int kAttnWin = 1024;    // entries whose slots and visibility are staged at a time
constexpr float kProbScale = 4096.f;

struct AttnView {
  const long long* acc;     // q|k|v sums [16][acc_ld] (fixed point), GPU row order
  int acc_ld;
  const float2* rope;       // [max_position][d/2]
  uint16_t* kpool;          // layer 0; layer l at + l * layer_stride
  uint16_t* vpool;
  size_t layer_stride;
  int cap, Hq, Hkv, d;
  float* part;              // [request][kv head][chunk][query][d + 4], AttnPlan::part0
  const int* cnt_kv;        // q|k|v units finished per kv head
  int kv_units;             // units per kv head when its q|k|v rows are complete
  const int* bt;            // beam table (entry -> physical slot) of this step
  const uint8_t* mask;
  int mask_stride;
  int packed;               // a mask row per token of request 0 instead of one per request
  uint32_t limit;
  uint16_t* out;
  int out_ld;
};

// A quotient in code that runs once per launch: inlined divisions are a good part
// of such code, and fetching it is what it costs.
__device__ __noinline__ unsigned quotient(unsigned a, unsigned b) { return a / b; }
__device__ __forceinline__ int n_chunks_of(int L, int cs) { return (int)quotient(L + cs - 1, cs); }

// Entries per chunk of a row of L entries: a function of the row alone.  (A row's
// entries times kv heads fit 32 bits: the pool holds 256 bytes or more for each.)
__device__ __forceinline__ int chunk_entries(int L, int Hkv, int grid) {
  int cs = max(kAttnChunkMin, (int)(quotient((unsigned)L * Hkv + grid - 1, grid) + 15) / 16 * 16);
  // rounding up can need a little more than the even share
  while (cs < L && Hkv * n_chunks_of(L, cs) > grid) cs += 16 * max(1, cs / 256);
  return min(cs, L);
}

// The attention of a step of several requests: filled by one warp, lane b for request b.
struct AttnPlan {
  int cs[kMaxRequests];     // entries per chunk of a request,
  int run[kMaxRequests];    // chunks per unit,
  int unit0[kMaxRequests];  // its first unit,
  int part0[kMaxRequests];  // and its first partial (rows of several chunks have them)
};

// Sum of v over the lanes before this one.
__device__ __forceinline__ int lanes_before(int v, int lane) {
  int t = v;
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += u;
  }
  return t - v;
}

// Runs grow from the even share of all entries until every unit finds a CTA, or
// are whole rows.  Returns the number of units.
__device__ __forceinline__ int attn_plan(const StepParams* sp, int G, int Hkv, int grid, int lane, AttnPlan* plan) {
  const unsigned all = 0xffffffffu;
  const bool mine = lane < sp->B;
  const int L = mine ? sp->req_len[lane] : 0;
  const int cs = mine ? chunk_entries(L, Hkv, grid) : 1, nc = mine ? n_chunks_of(L, cs) : 0;
  int share = max(kAttnChunkMin, (int)quotient((unsigned)__reduce_add_sync(all, L) * Hkv + grid - 1, grid));
  int run, units, total;
#pragma unroll 1
  for (;;) {
    run = min(max((int)quotient(share, cs), 1), nc);
    units = mine ? Hkv * n_chunks_of(nc, run) : 0;
    total = __reduce_add_sync(all, units);
    if (total <= grid || __all_sync(all, run == nc)) break;
    share += 16 * max(1, share / 256);
  }
  const int unit0 = lanes_before(units, lane);
  const int queries = mine ? G * (sp->req_tok0[lane + 1] - sp->req_tok0[lane]) : 0;
  const int part0 = lanes_before(nc > 1 ? Hkv * nc * queries : 0, lane);
  if (mine) {
    plan->cs[lane] = cs;
    plan->run[lane] = run;
    plan->unit0[lane] = unit0;
    plan->part0[lane] = part0;
  }
  __syncwarp();
  return total;
}

// Shared-memory layout of a unit's attention.  Query rows are padded so that
// the two rows of a quarter-warp's 16-byte loads fall on different banks.
template <int DPL>
struct AttnSmem {
  static constexpr int d = 32 * DPL;
  static constexpr int kQld = d + 32;                             // halves
  static constexpr size_t kQ = (size_t)kAttnQ * kQld * 2;         // fp16 queries, and the same for their remainders
  static constexpr size_t kRows = (size_t)kAttnWin * 4;           // pool row of each entry
  static constexpr size_t kVis = (size_t)kAttnWin * 2;            // bit t: token t sees the entry
  static constexpr size_t kScale = (size_t)kAttnQ * 4;            // score scale of each query
  static constexpr size_t kLoop = 2 * kQ + kRows + kVis + kScale;
  // the same space, once a chunk's entries are done: a tile's pieces of every warp
  static constexpr int kOld = part_stride(d);                     // floats per query of a piece
  static constexpr size_t kPieces = (size_t)kWarps * 8 * kOld * 4;
  static constexpr size_t kMl = (size_t)kWarps * 8 * 8;           // (max, sum) per piece and query
  static constexpr size_t kBytes = kLoop > kPieces + kMl ? kLoop : kPieces + kMl;
};

// Row of the q|k|v projection holding dimension i (< d/2) of q head h, or of
// k head h when `first` is the first k row; dimension i + d/2 is 8 rows
// further (kernels.h: rotary pairs share a 16-row tile).
__device__ __forceinline__ int rot_row(int first, int h, int i, int d) {
  return first + 16 * (h * (d >> 4) + (i >> 3)) + (i & 7);
}

// Queries q0 .. q0 + qn of a unit into shared memory: a warp per query reads
// the fixed-point q sums of the query's head and token, rotates them by the
// token's position (RoPE, pairs (i, i + d/2)), scales the row by a power of
// two and splits it into fp16 and the fp16 of what that left out.
template <int DPL>
__device__ __forceinline__ void attn_load_queries(const AttnView& a, const StepParams* sp, int hk, int tok0, int q0,
                                                  int qn, uint16_t* qhi, uint16_t* qlo, float* qscale) {
  constexpr int d = 32 * DPL, half = d / 2, kPair = half / 32, kRowsAtOnce = 4;
  const int G = a.Hq / a.Hkv, tid = opaque(threadIdx.x), warp = tid >> 5, lane = tid & 31;
  const float sm = rsqrtf(static_cast<float>(d));
  for (int b0 = warp; b0 < qn; b0 += kWarps * kRowsAtOnce) {
    long long lo[kRowsAtOnce][kPair], hi[kRowsAtOnce][kPair];
    float2 cs[kRowsAtOnce][kPair];
#pragma unroll
    for (int r = 0; r < kRowsAtOnce; ++r) {
      const int q = q0 + min(b0 + r * kWarps, qn - 1);
      const int m = tok0 + q / G, h = hk * G + q % G;
      const long long* row = a.acc + (size_t)m * a.acc_ld;
#pragma unroll
      for (int p = 0; p < kPair; ++p) {
        const int i = lane + 32 * p, R = rot_row(0, h, i, d);
        lo[r][p] = __ldcg(row + R);
        hi[r][p] = __ldcg(row + R + 8);
        cs[r][p] = a.rope[(size_t)sp->tok_pos[m] * half + i];
      }
    }
#pragma unroll
    for (int r = 0; r < kRowsAtOnce; ++r) {
      const int qi = b0 + r * kWarps;
      if (qi >= qn) break;
      float x[2 * kPair];
      uint32_t big = 0;
#pragma unroll
      for (int p = 0; p < kPair; ++p) {
        const float l = fixed_to_f32(lo[r][p]), h = fixed_to_f32(hi[r][p]);
        x[2 * p] = l * cs[r][p].x - h * cs[r][p].y;
        x[2 * p + 1] = h * cs[r][p].x + l * cs[r][p].y;
        big = max(big, max(__float_as_uint(fabsf(x[2 * p])), __float_as_uint(fabsf(x[2 * p + 1]))));
      }
      // 2^-e for the largest value's exponent e (the sums are below 2^32)
      const int e = max((int)(__reduce_max_sync(0xffffffffu, big) >> 23), 64);
      const float down = __uint_as_float((uint32_t)(254 - e) << 23);
      if (lane == 0) qscale[qi] = sm * __uint_as_float((uint32_t)e << 23);
      uint16_t* oh = qhi + (size_t)qi * AttnSmem<DPL>::kQld;
      uint16_t* ol = qlo + (size_t)qi * AttnSmem<DPL>::kQld;
#pragma unroll
      for (int p = 0; p < 2 * kPair; ++p) {
        const int i = lane + 32 * (p >> 1) + (p & 1) * half;
        const float v = x[p] * down;
        const uint16_t hv = f2h(v);
        oh[i] = hv;
        ol[i] = f2h(v - h2f(hv));
      }
    }
  }
}

// Merge of one (request, kv head, query): chunks in order, kMergeBatch at a
// time with all their loads in flight; lane c of a batch holds chunk c's max
// and sum, each lane DPL output dims.  The running result is rescaled when a
// batch raises the maximum (online softmax).  `base`: chunk 0's partial of
// this query; cstride floats between chunks.
template <int DPL>
__device__ __forceinline__ void attn_merge_warp(const float* base, size_t cstride, int nc, uint16_t* out, int lane) {
  constexpr int kMergeBatch = 16;
  using VecT = typename std::conditional<DPL == 4, float4, float2>::type;
  float M = -INFINITY, den = 0.f, num[DPL];
#pragma unroll
  for (int u = 0; u < DPL; ++u) num[u] = 0.f;
  for (int c0 = 0; c0 < nc; c0 += kMergeBatch) {
    float mc = -INFINITY, lc = 0.f;
    if (lane < kMergeBatch && c0 + lane < nc) {
      const float2 ml = __ldcg(reinterpret_cast<const float2*>(base + (size_t)(c0 + lane) * cstride));
      mc = ml.x;
      lc = ml.y;
    }
    VecT ov[kMergeBatch];
#pragma unroll
    for (int u = 0; u < kMergeBatch; ++u) {
      if (c0 + u < nc) {
        ov[u] = __ldcg(reinterpret_cast<const VecT*>(base + (size_t)(c0 + u) * cstride + 4) + lane);
      } else {
        ov[u] = VecT{};
      }
    }
    float bm = mc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, o));
    const float Mn = fmaxf(M, bm);
    const float alpha = (M == -INFINITY) ? 0.f : expf(M - Mn);
    den *= alpha;
#pragma unroll
    for (int u = 0; u < DPL; ++u) num[u] *= alpha;
    const float wl = (mc == -INFINITY) ? 0.f : expf(mc - Mn);
    float dl = lc * wl;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    den += dl;
#pragma unroll
    for (int u = 0; u < kMergeBatch; ++u) {
      const float w = __shfl_sync(0xffffffffu, wl, u);
      const float* f = reinterpret_cast<const float*>(&ov[u]);
#pragma unroll
      for (int v = 0; v < DPL; ++v) num[v] = fmaf(f[v], w, num[v]);
    }
    M = Mn;
  }
#pragma unroll
  for (int u = 0; u < DPL; ++u) out[DPL * lane + u] = f2h(num[u] / den);
}

// Partials (queries x chunks) up to which the last chunk's CTA merges alone: it
// saves the other CTAs' polls, but reads them all through one SM (528 bytes each
// at d = 128; 64 of them are one batch of loads per warp).
constexpr int kMergeAlone = 64;

// attn_run's warps share the area with their scores: below this many (chunks of more
// than 16 blocks for one query tile, of more than 11 for three) a unit goes chunk by
// chunk.  Layer 0's attention at 8B width, run / chunk by chunk: 4 rows of 2000
// entries 20 / 37 us, of 3500 (6 warps) 33 / 48, of 4300 (5) 63 / 58, of 5500 (4)
// 78 / 61, of 7500 (3) 140 / 76; 3 rows of 5 tokens on 2000 (8) 31 / 49, on 3000 (5)
// 45 / 48, on 5000 (3) 128 / 83.
constexpr int kRunWarps = 5;

// A CTA's unit, laid out once per launch (by one thread) for all layers.
struct AttnUnit {
  int total;                // the step's units
  int hk, tok0, nb, Q, P;
  int row;                  // of the mask and the beam table
  int cs, nc, c0, c1;       // entries per chunk, chunks of the row, this unit's
  int end;                  // the entry after the row's last
  int u, units;             // its place among the units of its (request, kv head)
  int part0;                // the (request, kv head)'s first partial
  int* cnt;                 // finished chunks of the (request, kv head)
  // attn_run, for units of several chunks (warps = 0: chunk by chunk, attn_chunk)
  int warps;                // that take part
  uint32_t qlo, rows;       // byte offsets in the area
};

// A step of one request: every chunk is a unit.
__device__ __forceinline__ void attn_one_row(const StepParams& sp, int Hkv, int grid, AttnUnit& n) {
  n.cs = chunk_entries(sp.req_len[0], Hkv, grid);
  n.nc = n_chunks_of(sp.req_len[0], n.cs);
  n.total = Hkv * n.nc;
}

template <int DPL, bool kMany>
__device__ __noinline__ void attn_unit_init(const AttnPlan& plan, const StepParams& sp, int G, int Hkv, int* cnt,
                                            uint32_t area_bytes, int unit, AttnUnit& n) {
  using S = AttnSmem<DPL>;
  int b = 0, run = 1, part0 = 0;
  if (kMany) {
    b = sp.B - 1;
#pragma unroll 1
    while (plan.unit0[b] > unit) --b;
    unit -= plan.unit0[b];
    run = plan.run[b];
    part0 = plan.part0[b];
    n.cs = plan.cs[b];
    n.nc = n_chunks_of(sp.req_len[b], n.cs);
  }
  const int units = kMany ? n_chunks_of(n.nc, run) : n.nc, hk = (int)quotient(unit, units);
  const int u = unit - hk * units, nb = sp.req_tok0[b + 1] - sp.req_tok0[b], Q = nb * G;
  n.row = b;
  n.hk = hk;
  n.tok0 = sp.req_tok0[b];
  n.nb = nb;
  n.Q = Q;
  n.P = sp.req_P[b];
  n.end = sp.req_len[b];
  n.u = u;
  n.units = units;
  n.c0 = u * run;
  n.c1 = min(n.c0 + run, n.nc);
  n.part0 = part0 + hk * n.nc * Q;
  n.cnt = cnt + b * Hkv + hk;
  if (kMany) {
    // a warp's scores take 512 bytes a block of its chunk, behind the queries and the entries' rows
    const int nqt = (Q + 7) >> 3, nblk = (n.cs + 15) >> 4;
    n.qlo = nqt * 8 * S::kQld * 2;
    n.rows = 2 * n.qlo;
    const int room = (int)area_bytes - (int)n.rows - (int)(S::kRows + S::kVis + S::kScale);
    const int fit = room > 0 ? min((int)quotient(room, 512 * nblk), kWarps) : 0;
    n.warps = n.c1 - n.c0 > 1 && Q <= kAttnQ && n.cs <= kAttnWin && fit >= kRunWarps ? fit : 0;
  }
}

// K rows of block blk: entries gid and gid + 8; a lane's share of each is d / 4 values.
template <int DPL>
__device__ __forceinline__ void attn_load_k(uint4 (&kf)[2][DPL], const uint16_t* kpool, const uint32_t* rows_s, int blk,
                                            int gid, int tig) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint4* p = reinterpret_cast<const uint4*>(kpool + (size_t)rows_s[16 * blk + 8 * i + gid] * (32 * DPL)) + tig;
#pragma unroll
    for (int j = 0; j < DPL; ++j) kf[i][j] = p[4 * j];
  }
}

// V rows of block blk: entries 2 tig, + 1, + 8, + 9; a lane's share of each is d / 8 values.
template <int DPL>
__device__ __forceinline__ void attn_load_v(uint4 (&vf)[4][DPL / 2], const uint16_t* vpool, const uint32_t* rows_s,
                                            int blk, int gid, int tig) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint4* p = reinterpret_cast<const uint4*>(
                         vpool + (size_t)rows_s[16 * blk + 8 * (r >> 1) + 2 * tig + (r & 1)] * (32 * DPL)) + gid;
#pragma unroll
    for (int j = 0; j < DPL / 2; ++j) vf[r][j] = p[8 * j];
  }
}

// Scores of query gid (qh, ql: its values and their remainders; qs: its scale, tk:
// its token) and entries 2 tig, + 1, + 8, + 9 of a block, -inf where it does not
// see them (vis: the block's bits).
template <int DPL>
__device__ __forceinline__ void attn_scores(float (&x)[4], const uint4 (&kf)[2][DPL], const uint16_t* qh,
                                            const uint16_t* ql, const uint16_t* vis, int tk, float qs, int tig) {
  const uint32_t va = *reinterpret_cast<const uint32_t*>(vis + 2 * tig) >> tk;
  const uint32_t vb = *reinterpret_cast<const uint32_t*>(vis + 8 + 2 * tig) >> tk;
  float s[2][2][4];  // two chains per 8 entries
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int e = 0; e < 2; ++e) s[i][e][0] = s[i][e][1] = s[i][e][2] = s[i][e][3] = 0.f;
#pragma unroll
  for (int j = 0; j < DPL; ++j) {
    const uint4 h = *reinterpret_cast<const uint4*>(qh + 32 * j);
    const uint4 l = *reinterpret_cast<const uint4*>(ql + 32 * j);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mma_16816(s[i][0], h.x, l.x, h.y, l.y, kf[i][j].x, kf[i][j].y);
      mma_16816(s[i][1], h.z, l.z, h.w, l.w, kf[i][j].z, kf[i][j].w);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float (&u)[2][4] = s[i >> 1];
    const int e = i & 1;
    const bool see = ((i < 2 ? va : vb) >> (16 * e)) & 1u;
    const float hi = u[0][e] + u[1][e], lo = u[0][2 + e] + u[1][2 + e];
    // (an infinite key: the remainders' product has a sign of its own, or none)
    x[i] = see ? (fabsf(hi) < INFINITY ? hi + lo : hi) * qs : -INFINITY;
  }
}

__device__ __forceinline__ float attn_block_max(const float (&x)[4]) {
  float mn = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
  mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
  return fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
}

// A block's probabilities and value sum into the running (mx, den, o): online softmax.
template <int DPL>
__device__ __forceinline__ void attn_values(const float (&x)[4], const uint4 (&vf)[4][DPL / 2], float (&o)[2 * DPL][4],
                                            float& mx, float& den, int tig) {
  const float mn = fmaxf(attn_block_max(x), mx);
  if (__any_sync(0xffffffffu, mn > mx)) {
    const float alpha = mx == -INFINITY ? 0.f : expf(mx - mn);
    den *= alpha;
    const float a0 = __shfl_sync(0xffffffffu, alpha, 8 * tig), a1 = __shfl_sync(0xffffffffu, alpha, 8 * tig + 4);
#pragma unroll
    for (int i = 0; i < 2 * DPL; ++i) {
      o[i][0] *= a0;
      o[i][1] *= a1;
      o[i][2] *= a0;
      o[i][3] *= a1;
    }
    mx = mn;
  }
  uint32_t ph[2], pl[2];  // the probabilities as the value sum's B fragments
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float p0 = x[2 * i] == -INFINITY ? 0.f : expf(x[2 * i] - mn) * kProbScale;
    const float p1 = x[2 * i + 1] == -INFINITY ? 0.f : expf(x[2 * i + 1] - mn) * kProbScale;
    den += p0 + p1;
    const uint16_t u = f2h(p0), w = f2h(p1);
    ph[i] = (uint32_t)u | ((uint32_t)w << 16);
    pl[i] = pack_h2(p0 - h2f(u), p1 - h2f(w));
  }
  // O^T += V^T P^T: a lane's 32-bit word u of the four entries' rows
  // holds dims 2 u and 2 u + 1 of its 8: rows gid and gid + 8 of a tile
#pragma unroll
  for (int i = 0; i < 2 * DPL; ++i) {
    const int j = i >> 2, u = i & 3;
    auto word = [&](const uint4& v) { return u == 0 ? v.x : u == 1 ? v.y : u == 2 ? v.z : v.w; };
    const uint32_t r0 = word(vf[0][j]), r1 = word(vf[1][j]), r2 = word(vf[2][j]), r3 = word(vf[3][j]);
    const uint32_t f0 = prmt_u32(r0, r1, 0x5410u), f1 = prmt_u32(r0, r1, 0x7632u);
    const uint32_t f2 = prmt_u32(r2, r3, 0x5410u), f3 = prmt_u32(r2, r3, 0x7632u);
    mma_16816(o[i], f0, f1, f2, f3, ph[0], ph[1]);
    mma_16816(o[i], f0, f1, f2, f3, pl[0], pl[1]);
  }
}

// Query 2 tig + e of a tile's value sums, as a lane holds them: 8 values of each 64 from 8 gid on.
template <int DPL>
__device__ __forceinline__ void attn_store_o(float* row, const float (&o)[2 * DPL][4], int e, int gid) {
#pragma unroll
  for (int j = 0; j < DPL / 2; ++j) {
    *reinterpret_cast<float4*>(row + 8 * gid + 64 * j) =
        make_float4(o[4 * j][e], o[4 * j][2 + e], o[4 * j + 1][e], o[4 * j + 1][2 + e]);
    *reinterpret_cast<float4*>(row + 8 * gid + 64 * j + 4) =
        make_float4(o[4 * j + 2][e], o[4 * j + 2][2 + e], o[4 * j + 3][e], o[4 * j + 3][2 + e]);
  }
}

// Entries j0 .. j0 + nw of the unit's row: their pool rows and visibility (bit t:
// token t sees the entry); entries that fill up the last block repeat the last one
// and are seen by nobody.
__device__ __forceinline__ void attn_stage(const AttnView& a, const AttnUnit& n, int j0, int nw, uint32_t* rows_s,
                                           uint16_t* vis_s, int tid) {
  const int P = n.P, nb = n.nb, hk = n.hk, row = n.row;
  for (int e = tid; e < (nw + 15) / 16 * 16; e += kThreads) {
    const int j = j0 + min(e, nw - 1);
    const int slot = __ldcg(a.bt + (size_t)row * a.cap + j);
    uint32_t bits = 0;
    if (e < nw) {
      if (a.packed) {  // a mask row per token, and no causal bound of its own
        const uint8_t* mp = a.mask + (size_t)n.tok0 * a.mask_stride + j;
#pragma unroll 4
        for (int t = 0; t < nb; ++t) bits |= (__ldcg(mp + (size_t)t * a.mask_stride) != 0 ? 1u : 0u) << t;
      } else if (__ldcg(a.mask + (size_t)row * a.mask_stride + j) != 0) {
        bits = 0xFFFFu << max(j - P, 0);  // token t sees entries up to P + t
      }
    }
    const uint32_t pr = (uint32_t)slot / (uint32_t)a.cap;
    rows_s[e] = (pr * a.Hkv + hk) * (uint32_t)a.cap + ((uint32_t)slot - pr * (uint32_t)a.cap);
    vis_s[e] = (uint16_t)bits;
  }
}

// Of entries j0 .. j0 + nj, the ones this step appends (they lie in the row's last
// chunks): k rotated by its token's position, both rounded to fp16.
template <int DPL>
__device__ __forceinline__ void attn_append(const AttnView& a, const AttnUnit& n, const StepParams* sp, int j0, int nj,
                                            uint16_t* kpool, uint16_t* vpool, int tid) {
  constexpr int d = 32 * DPL, half = d / 2;
  const int P = n.P, hk = n.hk, tok0 = n.tok0;
  const int r0 = max(P - j0, 0), nnew = nj - r0;
  if (nnew <= 0) return;
  const int k_first = a.Hq * d, v_first = (a.Hq + a.Hkv) * d;
  for (int e = tid; e < nnew * d; e += kThreads) {
    const int r = e / d, i = e - r * d;
    const int m = tok0 + (j0 + r0 + r - P);
    const long long* row = a.acc + (size_t)m * a.acc_ld;
    const int sl = sp->tok_slot[m];
    const size_t at = (((size_t)(sl / a.cap) * a.Hkv + hk) * a.cap + sl % a.cap) * d;
    if (i < half) {
      const int R = rot_row(k_first, hk, i, d);
      const float lo = fixed_to_f32(__ldcg(row + R)), hi = fixed_to_f32(__ldcg(row + R + 8));
      const float2 cs = a.rope[(size_t)sp->tok_pos[m] * half + i];
      kpool[at + i] = f2h(lo * cs.x - hi * cs.y);
      kpool[at + half + i] = f2h(hi * cs.x + lo * cs.y);
    } else {
      const int i2 = 2 * (i - half);
      const long long* vr = row + v_first + hk * d + i2;
      *reinterpret_cast<uint32_t*>(vpool + at + i2) = pack_h2(fixed_to_f32(__ldcg(vr)), fixed_to_f32(__ldcg(vr + 1)));
    }
  }
}

// One chunk by the CTA: its partials, or the outputs of a row of
// one chunk.
template <int DPL>
__device__ __forceinline__ void attn_chunk(const AttnView& a, const AttnUnit& n, int c, int layer, const StepParams* sp,
                                           uint8_t* area, int* status) {
  using S = AttnSmem<DPL>;
  constexpr int d = S::d;
  uint16_t* kpool = a.kpool + (size_t)layer * a.layer_stride;
  uint16_t* vpool = a.vpool + (size_t)layer * a.layer_stride;
  uint16_t* qhi = reinterpret_cast<uint16_t*>(area);
  uint16_t* qlo = reinterpret_cast<uint16_t*>(area + S::kQ);
  uint32_t* rows_s = reinterpret_cast<uint32_t*>(area + 2 * S::kQ);
  uint16_t* vis_s = reinterpret_cast<uint16_t*>(area + 2 * S::kQ + S::kRows);
  float* qscale = reinterpret_cast<float*>(area + 2 * S::kQ + S::kRows + S::kVis);
  float* pieces = reinterpret_cast<float*>(area);
  float2* ml_s = reinterpret_cast<float2*>(area + S::kPieces);
  const int tid = opaque(threadIdx.x), warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int hk = n.hk, tok0 = n.tok0, P = n.P, Q = n.Q, nc = n.nc;
  const int G = a.Hq / a.Hkv;
  const int j0 = c * n.cs, nj = min(n.cs, n.end - j0);

  uint4 kf[2][DPL], vf[4][DPL / 2];
#pragma unroll
  for (int j = 0; j < DPL; ++j) kf[0][j] = kf[1][j] = make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int j = 0; j < DPL / 2; ++j) vf[0][j] = vf[1][j] = vf[2][j] = vf[3][j] = make_uint4(0, 0, 0, 0);

  for (int q0 = 0; q0 < Q; q0 += kAttnQ) {
    const int qn = min(kAttnQ, Q - q0), nqt = (qn + 7) >> 3;
    const int eg = kWarps / nqt;             // warps side by side over the entries
    const int qt = warp / eg, g = warp - qt * eg;
    const bool active = qt < nqt;
    const int tk = (q0 + min(8 * qt + gid, qn - 1)) / G;  // the token of query gid
    float o[2 * DPL][4], mx = -INFINITY, den = 0.f, qs = 0.f;
#pragma unroll
    for (int i = 0; i < 2 * DPL; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
    for (int w0 = 0; w0 < nj; w0 += kAttnWin) {
      const int nw = min(kAttnWin, nj - w0), nblk = (nw + 15) >> 4;
      const bool first = q0 == 0 && w0 == 0;
      bool have = false;
      if (w0 > 0) cbar();  // the previous window's entries are done
      if (first || nj > kAttnWin || q0 > 0)
        attn_stage(a, n, j0 + w0, nw, rows_s, vis_s, tid);  // (the pieces overwrote it between passes)
      if (first) {
        cbar();
        // a block of entries from earlier steps loads during the wait for q|k|v
        have = active && g < nblk && j0 + 16 * g + 16 <= P;
        if (have) {
          attn_load_k<DPL>(kf, kpool, rows_s, g, gid, tig);
          attn_load_v<DPL>(vf, vpool, rows_s, g, gid, tig);
        }
        if (tid == 0) wait_count(a.cnt_kv + hk, a.kv_units, status, a.limit);
        cbar();
        attn_append<DPL>(a, n, sp, j0, nj, kpool, vpool, tid);
      }
      if (w0 == 0) attn_load_queries<DPL>(a, sp, hk, tok0, q0, qn, qhi, qlo, qscale);
      cbar();
      if (!active) continue;
      if (w0 == 0) qs = qscale[min(8 * qt + gid, qn - 1)];
      if (!have && g < nblk) {
        attn_load_k<DPL>(kf, kpool, rows_s, g, gid, tig);
        attn_load_v<DPL>(vf, vpool, rows_s, g, gid, tig);
      }
      const uint16_t* qh = qhi + (8 * qt + gid) * S::kQld + 8 * tig;
      const uint16_t* ql = qlo + (8 * qt + gid) * S::kQld + 8 * tig;
      for (int blk = g; blk < nblk; blk += eg) {
        const bool more = blk + eg < nblk;
        float x[4];
        attn_scores<DPL>(x, kf, qh, ql, vis_s + 16 * blk, tk, qs, tig);
        if (more) attn_load_k<DPL>(kf, kpool, rows_s, blk + eg, gid, tig);
        attn_values<DPL>(x, vf, o, mx, den, tig);
        if (more) attn_load_v<DPL>(vf, vpool, rows_s, blk + eg, gid, tig);
      }
    }
    // the CTA's pieces through shared memory
    const int ngr = min(eg, (min(nj, kAttnWin) + 15) >> 4);  // warps of a tile that had entries
    cbar();
    if (active && g < ngr) {
      den += __shfl_xor_sync(0xffffffffu, den, 1);
      den += __shfl_xor_sync(0xffffffffu, den, 2);
      if (tig == 0) ml_s[warp * 8 + gid] = make_float2(mx, den);
#pragma unroll
      for (int e = 0; e < 2; ++e) attn_store_o<DPL>(pieces + (size_t)(warp * 8 + 2 * tig + e) * S::kOld, o, e, gid);
    }
    cbar();
    for (int i = tid; i < qn * (d / 4); i += kThreads) {
      const int f = i % (d / 4), qi = i / (d / 4), r = qi & 7, wa = (qi >> 3) * eg;
      float M = -INFINITY, D = 0.f;
      float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int w = wa; w < wa + ngr; ++w) M = fmaxf(M, ml_s[w * 8 + r].x);
      for (int w = wa; w < wa + ngr; ++w) {
        const float2 ml = ml_s[w * 8 + r];
        const float k = ml.x == -INFINITY ? 0.f : expf(ml.x - M);
        const float4 v = *reinterpret_cast<const float4*>(pieces + (size_t)(w * 8 + r) * S::kOld + 4 * f);
        D = fmaf(ml.y, k, D);
        num.x = fmaf(v.x, k, num.x);
        num.y = fmaf(v.y, k, num.y);
        num.z = fmaf(v.z, k, num.z);
        num.w = fmaf(v.w, k, num.w);
      }
      const int q = q0 + qi;
      if (nc == 1) {
        uint2 h;
        h.x = pack_h2(num.x / D, num.y / D);
        h.y = pack_h2(num.z / D, num.w / D);
        *reinterpret_cast<uint2*>(a.out + (size_t)(tok0 + q / G) * a.out_ld + (hk * G + q % G) * d + 4 * f) = h;
      } else {
        float* p = a.part + (size_t)(n.part0 + c * Q + q) * part_stride(d);
        if (f == 0) *reinterpret_cast<float2*>(p) = make_float2(M, D);
        *reinterpret_cast<float4*>(p + 4 + 4 * f) = num;
      }
    }
    cbar();  // the partials are written, and the area is free
  }
}

// The unit's chunks, each query tile of a chunk by one warp, with the arithmetic and
// the order of attn_chunk: first all blocks' scores, kept in shared memory, and their
// largest; then the values of one piece after the other (piece g: blocks g, g + eg, ..,
// what warp g of attn_chunk adds), each scaled and added as the pieces meet there.
// No barrier between chunks: eight rows of 640..1642 entries at 8B width take 30.5 us
// a layer (norm, q|k|v and attention), chunk by chunk 79.
template <int DPL>
__device__ __forceinline__ void attn_run(const AttnView& a, const AttnUnit& n, int layer, const StepParams* sp,
                                         uint8_t* area, int* status) {
  using S = AttnSmem<DPL>;
  constexpr int d = S::d;
  uint16_t* kpool = a.kpool + (size_t)layer * a.layer_stride;
  uint16_t* vpool = a.vpool + (size_t)layer * a.layer_stride;
  const int tid = opaque(threadIdx.x), warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int hk = n.hk, tok0 = n.tok0, P = n.P, Q = n.Q, cs = n.cs, c0 = n.c0, c1 = n.c1, end = n.end;
  const int G = a.Hq / a.Hkv, nqt = (Q + 7) >> 3, eg = kWarps / nqt;
  uint16_t* qhi = reinterpret_cast<uint16_t*>(area);
  uint16_t* qlo = reinterpret_cast<uint16_t*>(area + n.qlo);
  uint32_t* rows_s = reinterpret_cast<uint32_t*>(area + n.rows);
  uint16_t* vis_s = reinterpret_cast<uint16_t*>(rows_s + kAttnWin);
  float* qscale = reinterpret_cast<float*>(vis_s + kAttnWin);
  float4* xs = reinterpret_cast<float4*>(qscale + kAttnQ) + warp * (cs >> 4) * 32 + lane;  // [block][lane]
  uint4 kf[2][DPL], vf[4][DPL / 2];
#pragma unroll
  for (int j = 0; j < DPL; ++j) kf[0][j] = kf[1][j] = make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int j = 0; j < DPL / 2; ++j) vf[0][j] = vf[1][j] = vf[2][j] = vf[3][j] = make_uint4(0, 0, 0, 0);
  const int staged = kAttnWin / cs;  // chunks whose entries are staged together
  for (int ca = c0; ca < c1; ca += staged) {
    const int j0 = ca * cs, nj = min(min(ca + staged, c1) * cs, end) - j0;
    const int items = (min(ca + staged, c1) - ca) * nqt;  // (chunk, query tile), tiles of a chunk side by side
    bool have = false;
    if (ca > c0) cbar();  // the entries before are done
    attn_stage(a, n, j0, nj, rows_s, vis_s, tid);
    if (ca == c0) {
      cbar();
      // a first block of entries from earlier steps loads during the wait for q|k|v
      have = warp < min(items, n.warps) && (c0 + warp / nqt) * cs + 16 <= P;
      if (have) attn_load_k<DPL>(kf, kpool, rows_s, warp / nqt * (cs >> 4), gid, tig);
      if (tid == 0) wait_count(a.cnt_kv + hk, a.kv_units, status, a.limit);
      cbar();
      attn_append<DPL>(a, n, sp, c0 * cs, min(c1 * cs, end) - c0 * cs, kpool, vpool, tid);
      attn_load_queries<DPL>(a, sp, hk, tok0, 0, Q, qhi, qlo, qscale);
    }
    cbar();
    for (int it = warp; it < items && warp < n.warps; it += n.warps) {
      const int ci = it / nqt, qt = it - ci * nqt, b0 = ci * (cs >> 4);
      const int nblk = (min(cs, end - (ca + ci) * cs) + 15) >> 4;
      const int q = 8 * qt + gid, tk = min(q, Q - 1) / G;
      const float qs = qscale[min(q, Q - 1)];
      const uint16_t* qh = qhi + q * S::kQld + 8 * tig;
      const uint16_t* ql = qlo + q * S::kQld + 8 * tig;
      if (!have) attn_load_k<DPL>(kf, kpool, rows_s, b0, gid, tig);
      have = false;
      float M = -INFINITY, x[4];
      for (int i = 0; i < nblk; ++i) {
        attn_scores<DPL>(x, kf, qh, ql, vis_s + 16 * (b0 + i), tk, qs, tig);
        if (i + 1 < nblk)
          attn_load_k<DPL>(kf, kpool, rows_s, b0 + i + 1, gid, tig);
        else
          attn_load_v<DPL>(vf, vpool, rows_s, b0, gid, tig);
        xs[32 * i] = make_float4(x[0], x[1], x[2], x[3]);
        M = fmaxf(M, attn_block_max(x));
      }
      float num[2 * DPL][4], D = 0.f;
#pragma unroll
      for (int i = 0; i < 2 * DPL; ++i) num[i][0] = num[i][1] = num[i][2] = num[i][3] = 0.f;
      const int ngr = min(eg, nblk);
      for (int g = 0; g < ngr; ++g) {
        float o[2 * DPL][4], mx = -INFINITY, den = 0.f;
#pragma unroll
        for (int i = 0; i < 2 * DPL; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
        for (int blk = g; blk < nblk; blk += eg) {
          const float4 xv = xs[32 * blk];
          const float y[4] = {xv.x, xv.y, xv.z, xv.w};
          attn_values<DPL>(y, vf, o, mx, den, tig);
          const int next = blk + eg < nblk ? blk + eg : g + 1;
          if (blk + eg < nblk || g + 1 < ngr) attn_load_v<DPL>(vf, vpool, rows_s, b0 + next, gid, tig);
        }
        den += __shfl_xor_sync(0xffffffffu, den, 1);
        den += __shfl_xor_sync(0xffffffffu, den, 2);
        const float k = mx == -INFINITY ? 0.f : expf(mx - M);
        D = fmaf(den, k, D);
        const float k0 = __shfl_sync(0xffffffffu, k, 8 * tig), k1 = __shfl_sync(0xffffffffu, k, 8 * tig + 4);
#pragma unroll
        for (int i = 0; i < 2 * DPL; ++i) {
          num[i][0] = fmaf(o[i][0], k0, num[i][0]);
          num[i][1] = fmaf(o[i][1], k1, num[i][1]);
          num[i][2] = fmaf(o[i][2], k0, num[i][2]);
          num[i][3] = fmaf(o[i][3], k1, num[i][3]);
        }
      }
      float* p = a.part + (size_t)(n.part0 + (ca + ci) * Q) * part_stride(d);
      if (tig == 0 && q < Q) *reinterpret_cast<float2*>(p + q * part_stride(d)) = make_float2(M, D);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int qe = 8 * qt + 2 * tig + e;
        if (qe < Q) attn_store_o<DPL>(p + qe * part_stride(d) + 4, num, e, gid);
      }
    }
  }
  cbar();  // the partials are written, and the area is free
}

// The row's outputs once all its chunks' partials are there.
template <int DPL>
__device__ __forceinline__ void attn_merge(const AttnView& a, const AttnUnit& n, int* status) {
  constexpr int d = 32 * DPL;
  const int tid = opaque(threadIdx.x), warp = tid >> 5, lane = tid & 31;
  const int Q = n.Q, G = a.Hq / a.Hkv;
  __shared__ int s_last;
  const bool alone = Q * n.nc <= kMergeAlone;
  if (tid == 0) {
    const int mine = n.c1 - n.c0;
    if (alone) {
      s_last = atom_add_acq_rel(n.cnt, mine) == n.nc - mine;
    } else {
      red_release_add_s32(n.cnt, mine);
      wait_count(n.cnt, n.nc, status, a.limit);
      s_last = 1;
    }
  }
  cbar();
  if (!s_last) return;
  const float* base = a.part + (size_t)n.part0 * part_stride(d);
  for (int q = alone ? warp : n.u + n.units * warp; q < Q; q += alone ? kWarps : n.units * kWarps)
    attn_merge_warp<DPL>(base + (size_t)q * part_stride(d), (size_t)Q * part_stride(d), n.nc,
                         a.out + (size_t)(n.tok0 + q / G) * a.out_ld + (n.hk * G + q % G) * d, lane);
}

template <int NT, int GPU, int DPL, bool kMany>
__global__ void __launch_bounds__(kThreads, 1) step_kernel(const __grid_constant__ StepKernelArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ GemvPhase s_gp[4];            // per projection kind: q|k|v, o, gate|up, down
  constexpr int kSlots = Geom<GPU>::kStepSlots;
  __shared__ AttnView s_av;
  __shared__ AttnPlan s_plan;              // (kMany)
  __shared__ AttnUnit s_unit;              // this CTA's attention unit
  __shared__ uint64_t s_nbar;              // the staged RMSNorm's bulk copies
  __shared__ StepParams s_sp;
  __shared__ const uint16_t* s_rowp[kMaxTokens];  // the step's fp16 input rows
  using SS = StepSmem<GPU>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* rings = smem;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + SS::kRing);
  uint8_t* att_area = smem + SS::area(a.L, a.gu_part, a.pro.M);
  static_assert(AttnSmem<DPL>::kBytes <= kAttnArea, "attention area too small");
  OpDesc* s_ops = reinterpret_cast<OpDesc*>(smem + SS::kOps);
  for (int i = threadIdx.x; i < 4 * a.L; i += kThreads) s_ops[i] = a.ops[i];
  if (threadIdx.x == 0) {
    mbar_init(&s_nbar, 1);
    ring_init_barriers(full, kWarps * kSlots);  // ends with the barrier-init fence
    if (blockIdx.x == 0) a.phase_clock[0] = globaltimer();
  }
  const auto plan = [&](int l) {
    if (kMany) {
      const int total = attn_plan(&s_sp, a.Hq / a.Hkv, a.Hkv, gridDim.x, l, &s_plan);
      if (l == 0) s_unit.total = total;
    } else if (l == 0) {
      attn_one_row(s_sp, a.Hkv, gridDim.x, s_unit);
    }
    if (l == 0 && (int)blockIdx.x < s_unit.total)
      attn_unit_init<DPL, kMany>(s_plan, s_sp, a.Hq / a.Hkv, a.Hkv, a.attn_cnt, a.area_bytes, blockIdx.x, s_unit);
  };
  prologue_params(a.pro, &s_sp, s_rowp, plan);  // ends with a block-wide barrier
  const int n_barriers = 4 * a.L + 1;
  if (s_sp.abort_step) {
    // every CTA sees the same inputs and rejects the step alike: count this
    // launch's barrier arrivals at once and write nothing
    if (threadIdx.x == 0) {
      red_release_add(a.barrier, (unsigned long long)n_barriers);
      if (blockIdx.x == 0) {
        atomicOr(a.pro.status, s_sp.abort_step & ~ST_STICKY);
        *reinterpret_cast<volatile int*>(a.status_out) = ld_acquire_s32(a.pro.status);
      }
    }
    return;
  }
  const StepParams* sp = &s_sp;
  const int M = sp->M;
  __shared__ GridBarrier gb;
  if (threadIdx.x == 0)
    gb = GridBarrier{a.barrier, a.barrier_base, a.status, a.phase_clock, 0, 0, a.debug_skip_arrival, a.wait_limit};
  // this warp's ring: its state stays in registers, except during attention,
  // which needs them all (s_ring holds it meanwhile)
  __shared__ WarpRing<GPU, kSlots> s_ring[kWarps];
  WarpRing<GPU, kSlots> ring;
  ring.ring = rings + (size_t)warp * kSlots * Geom<GPU>::kUnitBytes;
  ring.full = full + warp * kSlots;
  ring.n_used = 0;
  ring.timed_out = false;
  ring.start(s_ops, 4 * a.L, blockIdx.x * kWarps + warp, gridDim.x * kWarps, lane);
  // The normalised rows: in the area (idle during the q|k|v and gate|up
  // projections) when they fit, else read from act_h.
  const int xn_ld = xn_stride(a.H);
  const bool xn_smem = a.Kp_H == a.H && xn_bytes(a.H, M) <= a.area_bytes;
  uint16_t* xn = reinterpret_cast<uint16_t*>(att_area);
  // one row from the residual stream: staged through shared memory behind
  // the normalised row (rmsnorm_staged)
  const size_t stage_off = xn_bytes(a.H, 1);
  const bool norm_staged = M == 1 && xn_smem && a.H <= 24 * kThreads && stage_off + xn_stage_bytes(a.H, 1) <= a.area_bytes;
  long long* stage = reinterpret_cast<long long*>(att_area + stage_off);
  int norms_done = 0;
  uint32_t nphase = 0;
  const int G = a.Hq / a.Hkv;
  if (threadIdx.x < 4) {
    const int k = threadIdx.x;
    GemvPhase gp{};
    gp.act = k == 0 || k == 2 ? a.act_h : k == 1 ? a.act_attn : a.act_f;
    gp.act_ld = k == 0 || k == 2 ? a.Kp_H : k == 1 ? a.Kp_dq : a.Kp_F;
    gp.M = M;
    gp.act_s = (k == 0 || k == 2) && xn_smem ? smem_addr(att_area) : 0u;
    gp.act_s_ld = xn_ld;
    gp.status = a.status;
    gp.ep.kind = k == 0 ? EPI_QKV : k == 2 ? EPI_SWIGLU : EPI_RESID;
    gp.ep.dims = OpDims{k, a.Hq, a.Hkv, a.d, a.F, a.H};
    gp.ep.acc = k == 0 ? a.acc_qkv : k == 2 ? a.acc_gu : a.X;
    gp.ep.acc_ld = k == 0 ? (a.Hq + 2 * a.Hkv) * a.d : k == 2 ? s_ops[2].n_rb * kRowsPerBlock : a.H;
    gp.ep.cnt = k == 0 ? a.cnt_kv : k == 2 ? a.cnt_gu : nullptr;
    gp.ep.h = a.act_f;
    gp.ep.h_ld = a.Kp_F;
    gp.kv_rb_q = G * a.d / kRowsPerBlock;
    gp.kv_rb_per_head = a.d / kRowsPerBlock;
    gp.kv_rb_k = a.Hq * a.d / kRowsPerBlock;
    gp.kv_rb_v = (a.Hq + a.Hkv) * a.d / kRowsPerBlock;
    gp.part = reinterpret_cast<float*>(smem + SS::kOps + (size_t)4 * a.L * sizeof(OpDesc));
    s_gp[k] = gp;
  }
  if (threadIdx.x == 32) {
    AttnView av{};
    av.acc = a.acc_qkv;
    av.acc_ld = (a.Hq + 2 * a.Hkv) * a.d;
    av.rope = a.rope;
    av.kpool = a.kpool;
    av.vpool = a.vpool;
    av.layer_stride = a.layer_stride;
    av.cap = a.cap;
    av.Hq = a.Hq;
    av.Hkv = a.Hkv;
    av.d = a.d;
    av.part = a.attn_part;
    av.cnt_kv = a.cnt_kv;
    av.kv_units = (G + 2) * (a.d / kRowsPerBlock) * s_ops[0].upr;
    av.bt = a.pro.bt_dst;
    av.mask = a.mask;
    av.mask_stride = a.mask_stride;
    av.packed = a.packed;
    av.limit = a.wait_limit;
    av.out = a.act_attn;
    av.out_ld = a.Kp_dq;
    s_av = av;
  }
  prologue_work(a.pro, sp, s_rowp, a.X);
  cbar();
  gb.arrive();  // split barrier: waited for before the first attention

  const int g = blockIdx.x * kWarps + warp, nw = gridDim.x * kWarps;
  const int gt = blockIdx.x * kThreads + threadIdx.x, gs = gridDim.x * kThreads;
  const int qkv_rows = (a.Hq + 2 * a.Hkv) * a.d;

  // Phase k of layer l = ph / 4: q|k|v (k = 0), o, gate|up, down.  Every
  // phase body has one call site, so all of it is inlined into the kernel.
  for (int ph = 0; ph < 4 * a.L; ++ph) {
    const int l = ph >> 2, k = ph & 3;
    if (k == 0 || k == 2) {
      // RMSNorm of the attention (k = 0) or MLP block; before the first
      // layer from the step's input rows
      const uint16_t* nw_ = a.norms + (size_t)l * 2 * a.H + (k == 2 ? a.H : 0);
      if (norm_staged && ph != 0) {
        rmsnorm_staged(a.X, a.H, nw_, a.eps, xn, stage, &s_nbar, nphase, a.status);
      } else {
        // the one row of a staged step is fp16 here (8 KB): each CTA's own
        for (int m = norm_staged ? 0 : blockIdx.x; m < M; m += gridDim.x)
          rmsnorm_row(ph != 0, a.X, s_rowp, a.H, m, nw_, a.eps, norm_staged ? xn : a.act_h + (size_t)m * a.Kp_H,
                      norm_staged ? nullptr : a.norm_cnt);
      }
      if (!norm_staged) {
        norms_done += M;
        if (threadIdx.x == 0) wait_count(a.norm_cnt, norms_done, a.status, a.wait_limit);
        cbar();
        if (xn_smem) {
          // plain loads, all in flight: bulk copies cost a proxy fence and a
          // barrier wait more (8B width, 5 tokens, norm + gate|up 21.0 -> 18.4 us)
          constexpr int kAhead = 8;
          const int per = a.H / 8, pieces = M * per;  // of 16 bytes
          for (int e0 = threadIdx.x; e0 < pieces; e0 += kAhead * kThreads) {
            uint4 v[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
              const int e = e0 + i * kThreads, m = e / per;
              v[i] = e < pieces ? __ldcg(reinterpret_cast<const uint4*>(a.act_h + (size_t)m * a.Kp_H) + (e - m * per))
                                : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
              const int e = e0 + i * kThreads, m = e / per;
              if (e < pieces) *(reinterpret_cast<uint4*>(xn + (size_t)m * xn_ld) + (e - m * per)) = v[i];
            }
          }
          cbar();
        }
      }
    } else if (k == 1) {
      // the q|k|v sums and counts are consumed: clear them for the next layer
      for (int e = gt; e < M * qkv_rows; e += gs) __stcg(a.acc_qkv + e, 0LL);
      if (blockIdx.x == 0) {
        if (threadIdx.x < a.Hkv) __stcg(a.cnt_kv + threadIdx.x, 0);
        for (int e = threadIdx.x; e < sp->B * a.Hkv; e += kThreads) __stcg(a.attn_cnt + e, 0);
      }
    }
    gemv_run<NT, GPU, kSlots>(ring, &s_ops[ph], &s_gp[k], g, nw, lane);
    if (k == 0) {
      if (lane == 0) s_ring[warp] = ring;
      __syncwarp();
      if (l == 0) gb.wait();        // the prologue's tables and residual are complete
      else if (xn_smem) cbar();     // the attention reuses the normalised rows' space
      const int total = s_unit.total;
      for (int unit = blockIdx.x; unit < total; unit += gridDim.x) {
        if (total > (int)gridDim.x && (l > 0 || unit != (int)blockIdx.x)) {  // several units per CTA
          cbar();
          if (threadIdx.x == 0)
            attn_unit_init<DPL, kMany>(s_plan, s_sp, a.Hq / a.Hkv, a.Hkv, a.attn_cnt, a.area_bytes, unit, s_unit);
          cbar();
        }
        if (kMany && s_unit.warps > 0)
          attn_run<DPL>(s_av, s_unit, l, sp, att_area, a.status);
        else
          for (int c = s_unit.c0; c < (kMany ? s_unit.c1 : s_unit.c0 + 1); ++c)
            attn_chunk<DPL>(s_av, s_unit, c, l, sp, att_area, a.status);
        if (s_unit.nc > 1) attn_merge<DPL>(s_av, s_unit, a.status);
      }
      __syncwarp();
      asm volatile("" ::: "memory");
      ring = s_ring[warp];
    }
    gb.sync();
  }
  // hidden_out = fp16(x): one rounding from the exact fixed-point value
  for (int e = gt; e < M * a.H; e += gs) {
    const double v = static_cast<double>(__ldcg(a.X + e)) * kFixInv;
    a.pro.hidden_out[e] = __half_as_ushort(__double2half(v));
  }
  if (blockIdx.x == 0 && threadIdx.x < sp->B) a.pro.lens[threadIdx.x] = sp->req_len[threadIdx.x];
  if (ring.timed_out && lane == 0) atomicOr(a.status, ST_WAIT_TIMEOUT);
  // The last CTA to finish hands a nonzero status to the host-mapped mirror,
  // so no copy-engine transfer has to follow the step on the stream.
  cbar();
  if (threadIdx.x == 0 && atom_add_acq_rel(a.exit_count, 1) == (int)gridDim.x - 1) {
    *a.exit_count = 0;
    *a.norm_cnt = 0;
    const int st = ld_acquire_s32(a.status);
    if (st) *reinterpret_cast<volatile int*>(a.status_out) = st;
  }
}

template <int NT, int GPU, int DPL, bool kMany>
cudaError_t launch_t(const StepKernelArgs& a, int grid, cudaStream_t s) {
  auto kern = step_kernel<NT, GPU, DPL, kMany>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = StepSmem<GPU>::area(a.L, a.gu_part, a.pro.M) + a.area_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int NT, int GPU, int DPL, bool kMany>
size_t dyn_limit_t() {
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, step_kernel<NT, GPU, DPL, kMany>) != cudaSuccess) return 0;
  return (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
}

// The largest dynamic shared memory the kernel may take.
template <int NT, int GPU, int DPL, bool kMany>
cudaError_t setup_t() {
  return cudaFuncSetAttribute(step_kernel<NT, GPU, DPL, kMany>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)dyn_limit_t<NT, GPU, DPL, kMany>());
}

// Dynamic shared memory every kernel of a group size and head dim may take.
template <int GPU, int DPL>
size_t dyn_limit() {
  return std::min(std::min(dyn_limit_t<1, GPU, DPL, false>(), dyn_limit_t<1, GPU, DPL, true>()),
                  std::min(dyn_limit_t<2, GPU, DPL, false>(), dyn_limit_t<2, GPU, DPL, true>()));
}

// Bytes of the shared-memory area for steps of M tokens: room for the
// normalised rows where the kernel's limit allows it.
template <int GPU>
size_t area_bytes_t(int H, int L, bool part, int M, size_t limit) {
  const size_t want = xn_bytes(H, M) + xn_stage_bytes(H, M);
  if (want <= kAttnArea || StepSmem<GPU>::area(L, part, M) + want > limit) return kAttnArea;
  return want;
}

}  // namespace

int step_barriers(int n_layers) { return 4 * n_layers + 1; }

size_t step_dyn_limit(int group, int head_dim) {
  if (head_dim == 128) return group == 128 ? dyn_limit<1, 4>() : group == 64 ? dyn_limit<2, 4>() : dyn_limit<4, 4>();
  return group == 128 ? dyn_limit<1, 2>() : group == 64 ? dyn_limit<2, 2>() : dyn_limit<4, 2>();
}

bool step_gu_part_fits(int group, int L, size_t limit) {
  const size_t area = group == 128  ? StepSmem<1>::area(L, true, kMaxTokens)
                      : group == 64 ? StepSmem<2>::area(L, true, kMaxTokens)
                                    : StepSmem<4>::area(L, true, kMaxTokens);
  return area + kAttnArea <= limit;
}

size_t step_area_bytes(int group, int H, int L, bool part, int M, size_t limit) {
  if (group == 128) return area_bytes_t<1>(H, L, part, M, limit);
  if (group == 64) return area_bytes_t<2>(H, L, part, M, limit);
  return area_bytes_t<4>(H, L, part, M, limit);
}

int step_gu_split(int n_rb, int upr, int grid) {
  if (n_rb < 1 || upr < 1 || grid < 1) return 0;
  const long long nw = (long long)grid * kWarps;
  const long long even = ((long long)n_rb * upr + nw - 1) / nw;  // most units per warp, grid-wide split
  int best = 0;
  for (int q = 1; q <= kWarps; ++q) {
    if (kWarps % q != 0 || (long long)n_rb * q > nw) continue;  // one round of CTAs
    const long long most = (upr + q - 1) / q;
    if (most <= even + std::max(1LL, even / 16)) best = q;  // about as balanced as the grid-wide split
  }
  return best;
}

size_t step_attention_part_floats(int grid, int G, int d) {
  return (size_t)grid * (kMaxTokens * G) * part_stride(d);
}

cudaError_t step_setup(int group, int head_dim) {
  cudaError_t e = cudaSuccess;
#define SETUP_PAIR(GPU, DPL)                                              \
  if ((e = setup_t<1, GPU, DPL, false>()) != cudaSuccess) return e;       \
  if ((e = setup_t<1, GPU, DPL, true>()) != cudaSuccess) return e;        \
  if ((e = setup_t<2, GPU, DPL, false>()) != cudaSuccess) return e;       \
  if ((e = setup_t<2, GPU, DPL, true>()) != cudaSuccess) return e;
  if (head_dim == 128) {
    if (group == 128) { SETUP_PAIR(1, 4) }
    else if (group == 64) { SETUP_PAIR(2, 4) }
    else if (group == 32) { SETUP_PAIR(4, 4) }
  } else if (head_dim == 64) {
    if (group == 128) { SETUP_PAIR(1, 2) }
    else if (group == 64) { SETUP_PAIR(2, 2) }
    else if (group == 32) { SETUP_PAIR(4, 2) }
  } else {
    return cudaErrorInvalidValue;
  }
#undef SETUP_PAIR
  return e;
}

cudaError_t launch_step(const StepKernelArgs& a, int nt, int group, int grid, cudaStream_t s) {
  const int dpl = a.d / 32;
  const bool many = a.pro.B > 1;
#define LAUNCH(GPU, DPL)                                                                              \
  return nt == 1 ? (many ? launch_t<1, GPU, DPL, true>(a, grid, s) : launch_t<1, GPU, DPL, false>(a, grid, s)) \
                 : (many ? launch_t<2, GPU, DPL, true>(a, grid, s) : launch_t<2, GPU, DPL, false>(a, grid, s));
  if (dpl == 4) {
    if (group == 128) LAUNCH(1, 4)
    if (group == 64) LAUNCH(2, 4)
    if (group == 32) LAUNCH(4, 4)
  } else if (dpl == 2) {
    if (group == 128) LAUNCH(1, 2)
    if (group == 64) LAUNCH(2, 2)
    if (group == 32) LAUNCH(4, 2)
  }
#undef LAUNCH
  return cudaErrorInvalidValue;
}

}  // namespace shard
