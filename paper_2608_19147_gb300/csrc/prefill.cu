// Prefill: a prompt of S tokens through the stage in one call (Section 3.4:
// the stateful cache is filled by running the prompt through the shard).
// The arithmetic is the decode step's, for S new tokens of one request: the
// same rounding points (fp16 normalised activations, attention output,
// SwiGLU output, appended K/V and the output), causal attention among the new
// tokens and over the row's unmasked cache.  The projections are dense
// contractions here and run on the tensor cores (gemm_tc.cu), the attention on
// mma.sync over blocks of tokens (prefill_flash_kernel); the rest are small
// per-token kernels, launched layer by layer on the caller's stream.
// Each of a layer's eight kernels is launched behind the one before it
// (launch.cuh): its CTAs take their places, and a projection's also fill their
// rings of weights, while that one ends. It lets the next one come only after
// its own wait, so a kernel sees all kernels before it ended, not just the last.
// Bound otherwise by launch gaps of 1.5..2.5 us each: 4 layers at 8B width, 77
// tokens 704 -> 622 us, 512 tokens 1509 -> 1452.
#include <algorithm>

#include "common.cuh"
#include "launch.cuh"

namespace shard {
namespace {


// Device-side argument checks (values that live on the device): token ids in
// [0, vocab), positions in [0, max_position), the mask open at every new
// entry.  A violation sets a status bit; the host then reports the call as
// rejected and the caller must reset the row.
__global__ void prefill_check_kernel(const int* token_ids, int vocab, const int* pos, int max_position,
                                     const uint8_t* mask, int P, int S, int* status) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < S; t += gridDim.x * blockDim.x) {
    int bits = 0;
    if (token_ids) {
      const int tok = token_ids[t];
      if (tok < 0 || tok >= vocab) bits |= ST_TOKEN;
    }
    const int p = pos[t];
    if (p < 0 || p >= max_position) bits |= ST_POSITION;
    if (mask[P + t] == 0) bits |= ST_MASK_NEW;
    if (bits) atomicOr(status, bits);
  }
}

// v plus the parts of a projection's output behind y, in order; a fixed trip
// count, so that all parts' (and several callers') loads are in flight at once.
__device__ __forceinline__ float4 add_parts(float4 v, const float* y, size_t y_part, int first, int parts) {
  float4 u[kGemmMaxParts];
#pragma unroll
  for (int p = 0; p < kGemmMaxParts; ++p)
    if (p >= first) u[p] = p < parts ? *reinterpret_cast<const float4*>(y + p * y_part) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int p = 0; p < kGemmMaxParts; ++p)
    if (p >= first && p < parts) {
      v.x += u[p].x;
      v.y += u[p].y;
      v.z += u[p].z;
      v.w += u[p].w;
    }
  return v;
}

__global__ void set_int_kernel(int* p, int v) { *p = v; }

// One CTA per token: the residual x[t] (first the input row, later x[t] plus the
// parts of the projection before it), then act[t] = fp16(x r w) with
// r = 1 / sqrt(mean(x^2) + eps), or after the last layer out[t] = fp16(x).
// One pass over the row: kP pieces (float4) per thread stay in registers
// between the sum of squares and the scaling, the rest of a longer row is read
// back.  Bound by its L2 traffic (20 bytes per value with one part); residual
// add and norm apart moved 28 and took two launches.
constexpr int kNormThreads = 256;
__global__ void __launch_bounds__(kNormThreads) prefill_norm_kernel(const __grid_constant__ PrefillNormArgs a) {
  constexpr int kP = 8;
  __shared__ float s_part[kNormThreads / 32];
  const int t = blockIdx.x, tid = threadIdx.x, H4 = a.H / 4;
  pdl_wait();
  pdl_launch_dependents();
  float4* xr = reinterpret_cast<float4*>(a.x + (size_t)t * a.H);
  const uint16_t* in = nullptr;
  if (a.hidden_in) {
    in = a.hidden_in + (size_t)t * a.H;
  } else if (a.token_ids) {
    const int tok = __ldg(a.token_ids + t);  // out-of-range ids were flagged by the check; read a valid row
    in = a.embedding + (size_t)(tok < 0 || tok >= a.vocab ? 0 : tok) * a.H;
  }
  // the caller's buffers may be aligned to their values only
  const bool in8 = reinterpret_cast<uintptr_t>(in) % 8 == 0, out8 = reinterpret_cast<uintptr_t>(a.out) % 8 == 0;
  auto get = [&](int c) {
    if (in && !in8) return make_float4(h2f(in[4 * c]), h2f(in[4 * c + 1]), h2f(in[4 * c + 2]), h2f(in[4 * c + 3]));
    if (in) {
      const uint2 u = *reinterpret_cast<const uint2*>(in + 4 * c);
      return make_float4(h2f(u.x & 0xFFFFu), h2f(u.x >> 16), h2f(u.y & 0xFFFFu), h2f(u.y >> 16));
    }
    return add_parts(xr[c], a.y + (size_t)t * a.H + 4 * c, a.y_part, 0, a.parts);
  };
  auto halves = [](float4 v) {
    return make_uint2((uint32_t)f2h(v.x) | ((uint32_t)f2h(v.y) << 16), (uint32_t)f2h(v.z) | ((uint32_t)f2h(v.w) << 16));
  };
  if (!a.w) {
    for (int c = tid; c < H4; c += kNormThreads) {
      const uint2 u = halves(get(c));
      uint16_t* o = a.out + (size_t)t * a.H + 4 * c;
      if (out8) {
        *reinterpret_cast<uint2*>(o) = u;
      } else {
        o[0] = (uint16_t)u.x;
        o[1] = (uint16_t)(u.x >> 16);
        o[2] = (uint16_t)u.y;
        o[3] = (uint16_t)(u.y >> 16);
      }
    }
    return;
  }
  float4 v[kP];
  float ss = 0.f;
  if (in) {
#pragma unroll
    for (int i = 0; i < kP; ++i) {
      const int c = tid + i * kNormThreads;
      v[i] = c < H4 ? get(c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  } else {
#pragma unroll
    for (int i = 0; i < kP; ++i) {
      const int c = tid + i * kNormThreads;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < H4) v[i] = add_parts(xr[c], a.y + (size_t)t * a.H + 4 * c, a.y_part, 0, a.parts);
    }
  }
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kNormThreads;
    if (c < H4) xr[c] = v[i];
    ss += v[i].x * v[i].x + v[i].y * v[i].y + v[i].z * v[i].z + v[i].w * v[i].w;
  }
  for (int c = tid + kP * kNormThreads; c < H4; c += kNormThreads) {
    const float4 u = get(c);
    xr[c] = u;
    ss += u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w;
  }
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((tid & 31) == 0) s_part[tid >> 5] = ss;
  __syncthreads();
  float tsum = 0.f;
  for (int i = 0; i < kNormThreads / 32; ++i) tsum += s_part[i];
  const float r = rsqrtf(tsum / a.H + a.eps);
  auto emit = [&](int c, float4 x) {
    const uint2 u = *reinterpret_cast<const uint2*>(a.w + 4 * c);
    const int k = 4 * c;
    *reinterpret_cast<uint2*>(a.act + (size_t)t * a.act_ld + (k & ~31) + act_pos(k & 31)) =
        halves(make_float4(x.x * r * h2f(u.x & 0xFFFFu), x.y * r * h2f(u.x >> 16), x.z * r * h2f(u.y & 0xFFFFu),
                           x.w * r * h2f(u.y >> 16)));
  };
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const int c = tid + i * kNormThreads;
    if (c < H4) emit(c, v[i]);
  }
  for (int c = tid + kP * kNormThreads; c < H4; c += kNormThreads) emit(c, xr[c]);
}

// RoPE (pairs (i, i + d/2), the token's position) on q (kept in fp32) and k;
// k and v rounded to fp16 and appended to the pool at the row's next slots.
// Four dims per thread, the projection's parts added in order.
__global__ void __launch_bounds__(256) prefill_rope_append_kernel(const __grid_constant__ PrefillLayerArgs a) {
  const int d = a.d, half = d / 2, h4 = half / 4;
  const int rot = (a.Hq + a.Hkv) * h4, per_tok = rot + a.Hkv * d / 4;
  const int n = a.S * per_tok;
  pdl_wait();
  pdl_launch_dependents();
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int t = e / per_tok, r = e % per_tok;
    const float* yr = a.y + (size_t)t * a.y_ld;
    auto get = [&](int row) {
      return add_parts(*reinterpret_cast<const float4*>(yr + row), yr + row, a.y_part, 1, a.parts);
    };
    auto halves = [](float4 v) {
      return make_uint2((uint32_t)f2h(v.x) | ((uint32_t)f2h(v.y) << 16), (uint32_t)f2h(v.z) | ((uint32_t)f2h(v.w) << 16));
    };
    const size_t kv = (((size_t)a.row * a.Hkv) * a.cap + (size_t)(a.slot0 + t)) * d;  // head 0's entry of this token
    if (r < rot) {
      const int h = r / h4, i = 4 * (r % h4);
      const int p = __ldg(a.pos + t);
      const float4* cs = reinterpret_cast<const float4*>(
          a.rope + (size_t)(p < 0 || p >= a.max_position ? 0 : p) * half + i);  // out-of-range positions were flagged
      const float4 c0 = cs[0], c1 = cs[1];
      const float4 lo = get(h * d + i), hi = get(h * d + half + i);
      const float4 olo = make_float4(lo.x * c0.x - hi.x * c0.y, lo.y * c0.z - hi.y * c0.w, lo.z * c1.x - hi.z * c1.y,
                                     lo.w * c1.z - hi.w * c1.w);
      const float4 ohi = make_float4(hi.x * c0.x + lo.x * c0.y, hi.y * c0.z + lo.y * c0.w, hi.z * c1.x + lo.z * c1.y,
                                     hi.w * c1.z + lo.w * c1.w);
      if (h < a.Hq) {
        float* q = a.q + (size_t)t * a.Hq * d + h * d + i;
        *reinterpret_cast<float4*>(q) = olo;
        *reinterpret_cast<float4*>(q + half) = ohi;
      } else {
        uint16_t* kp = a.kpool + kv + (size_t)(h - a.Hq) * a.cap * d + i;
        *reinterpret_cast<uint2*>(kp) = halves(olo);
        *reinterpret_cast<uint2*>(kp + half) = halves(ohi);
      }
    } else {
      const int rv = 4 * (r - rot), h = rv / d, i = rv % d;
      *reinterpret_cast<uint2*>(a.vpool + kv + (size_t)h * a.cap * d + i) = halves(get((a.Hq + a.Hkv) * d + rv));
    }
  }
}

// Activations in natural order to act_pos order (the test export's input).
__global__ void act_order_kernel(const uint16_t* x, int x_ld, int S, int Kp, uint16_t* out, int out_ld) {
  const size_t n = (size_t)S * Kp / 4;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int t = (int)(e / (Kp / 4)), k = 4 * (int)(e % (Kp / 4));
    *reinterpret_cast<uint2*>(out + (size_t)t * out_ld + (k & ~31) + act_pos(k & 31)) =
        *reinterpret_cast<const uint2*>(x + (size_t)t * x_ld + k);
  }
}

// Causal attention of the new tokens on the tensor cores (mma.sync m16n8k16),
// one CTA per (block of 64 / G tokens, kv head hk, part of the cache), 4 warps:
// query row r of the 64 is token t0 + r / G, query head hk G + r % G, and warp w
// owns rows 16 w .. + 15, so every K/V tile is read once for all the block's
// queries. Tiles of 64 entries (a row that may be prefilled holds its entries
// contiguously) come into shared memory with asynchronous copies, one tile
// ahead. Scores S = Q K^T with Q split into fp16 hi + lo parts (together ~22
// bits of q, so the scores match an fp32 q); online softmax per row in fp32;
// O += P V with P split the same way; fp32 accumulators. Entry j is visible to
// token t iff j <= P + t and mask[j] != 0.
// The bound is the tensor pipe (256 MMAs per warp and tile, ~2000 cycles) once
// the copies run ahead, and the length of a CTA's chain of tiles when there
// are few blocks: the cache is then cut into parts (launch_attn_t), each CTA
// leaves (max, sum, unnormalised output) per row, and the last one of a block
// combines them in order.
// 8B width, per launch: 512 tokens 83 -> 47 us, 77 tokens on ~900 entries 209 -> 42
// (before: synchronous tile loads, one CTA per block for the whole cache).
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(const void* p, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_addr(p)));
}
// 16 bytes to shared memory, asynchronously; zeros if !take.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool take) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(take ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(const void* p, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_addr(p)));
}
// fp16x2 of (lo, hi) and the fp16x2 of what each rounding left out
__device__ __forceinline__ void split_h2(float lo, float hi, uint32_t& h, uint32_t& l) {
  const uint16_t a = f2h(lo), b = f2h(hi);
  h = (uint32_t)a | ((uint32_t)b << 16);
  l = (uint32_t)f2h(lo - h2f(a)) | ((uint32_t)f2h(hi - h2f(b)) << 16);
}

template <int D>
struct FlashSmem {
  static constexpr int kLd = D + 8;  // row stride (halves): 16-byte rows, conflict-free fragment reads
  uint16_t k[2][64][kLd], v[2][64][kLd];
  uint8_t vis[2][64];
};

template <int D, int G>
__global__ void __launch_bounds__(128) prefill_flash_kernel(const __grid_constant__ PrefillLayerArgs a) {
  constexpr int TB = 64 / G;  // tokens per CTA
  constexpr int KS = D / 16;  // k16 steps over the head dimension
  constexpr int ND = D / 8;   // n8 tiles over the head dimension
  extern __shared__ __align__(16) uint8_t flash_smem[];
  __shared__ int s_last;
  FlashSmem<D>& sm = *reinterpret_cast<FlashSmem<D>*>(flash_smem);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int t0 = blockIdx.x * TB, hk = blockIdx.y;
  const int P = a.P, S = a.S;
  const float scale = rsqrtf((float)D);
  const int last = P + min(t0 + TB, S) - 1;  // the block's last token's limit
  const int tiles = last / 64 + 1;
  const int tile0 = tiles * (int)blockIdx.z / (int)gridDim.z, tile1 = tiles * (int)(blockIdx.z + 1) / (int)gridDim.z;
  const uint16_t* kp = a.kpool + ((size_t)a.row * a.Hkv + hk) * a.cap * D;
  const uint16_t* vp = a.vpool + ((size_t)a.row * a.Hkv + hk) * a.cap * D;
  // Q rows as fp16 hi (in K's second buffer) and lo (in V's), then this warp's
  // fragments; the first tile's copies run meanwhile
  auto copy_tile = [&](int tile) {
    const int buf = (tile - tile0) & 1, j0 = 64 * tile;
    for (int e = tid; e < 64 * (D / 8); e += 128) {
      const int r = e / (D / 8), c = e % (D / 8);
      const bool take = j0 + r <= last;
      const size_t off = (size_t)(take ? j0 + r : 0) * D + 8 * c;
      cp_async16(&sm.k[buf][r][8 * c], kp + off, take);
      cp_async16(&sm.v[buf][r][8 * c], vp + off, take);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto mask_of = [&](int tile) -> uint8_t {  // of entry 64 tile + tid, for threads below 64
    const int j = 64 * tile + tid;
    return tid < 64 && j <= last ? __ldg(a.mask + j) : 0;
  };
  pdl_wait();
  pdl_launch_dependents();
  if (tile0 < tile1) copy_tile(tile0);
  uint8_t seen = tile0 < tile1 ? mask_of(tile0) : 0;
  for (int e = tid; e < 16 * D; e += 128) {
    const int r = 4 * e / D, c = 4 * e % D, t = t0 + r / G;
    const float4 v = t < S ? *reinterpret_cast<const float4*>(a.q + (size_t)t * a.Hq * D + (hk * G + r % G) * D + c)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t h0, l0, h1, l1;
    split_h2(v.x, v.y, h0, l0);
    split_h2(v.z, v.w, h1, l1);
    *reinterpret_cast<uint2*>(&sm.k[1][r][c]) = make_uint2(h0, h1);
    *reinterpret_cast<uint2*>(&sm.v[1][r][c]) = make_uint2(l0, l1);
  }
  __syncthreads();
  const int ra = 16 * warp + gid, rb = ra + 8;  // this thread's two query rows
  uint32_t qh[KS][4], ql[KS][4];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const int c = 16 * ks + 2 * tig;
    qh[ks][0] = *reinterpret_cast<const uint32_t*>(&sm.k[1][ra][c]);
    qh[ks][1] = *reinterpret_cast<const uint32_t*>(&sm.k[1][rb][c]);
    qh[ks][2] = *reinterpret_cast<const uint32_t*>(&sm.k[1][ra][c + 8]);
    qh[ks][3] = *reinterpret_cast<const uint32_t*>(&sm.k[1][rb][c + 8]);
    ql[ks][0] = *reinterpret_cast<const uint32_t*>(&sm.v[1][ra][c]);
    ql[ks][1] = *reinterpret_cast<const uint32_t*>(&sm.v[1][rb][c]);
    ql[ks][2] = *reinterpret_cast<const uint32_t*>(&sm.v[1][ra][c + 8]);
    ql[ks][3] = *reinterpret_cast<const uint32_t*>(&sm.v[1][rb][c + 8]);
  }
  const int tok_a = t0 + ra / G, tok_b = t0 + rb / G;
  const int lim_a = P + tok_a, lim_b = P + tok_b;  // causal limits
  float o[ND][4];
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
  float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
  for (int tile = tile0; tile < tile1; ++tile) {
    const int buf = (tile - tile0) & 1, j0 = 64 * tile;
    if (tid < 64) sm.vis[buf][tid] = seen;
    __syncthreads();  // the other buffer (the previous tile, or the Q staging) is read
    if (tile + 1 < tile1) {
      copy_tile(tile + 1);
      seen = mask_of(tile + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const uint16_t (*Ks)[FlashSmem<D>::kLd] = sm.k[buf], (*Vs)[FlashSmem<D>::kLd] = sm.v[buf];
    const uint8_t* vis = sm.vis[buf];
    float sc[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KS; ks += 2)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        uint32_t b0, b1, b2, b3;  // entries 8 nt .. + 7, inputs 16 ks .. + 31
        ldsm_x4(&Ks[8 * nt + (lane & 7)][16 * ks + 8 * (lane >> 3)], b0, b1, b2, b3);
        mma16816(sc[nt], qh[ks], b0, b1);
        mma16816(sc[nt], ql[ks], b0, b1);
        mma16816(sc[nt], qh[ks + 1], b2, b3);
        mma16816(sc[nt], ql[ks + 1], b2, b3);
      }
    // mask and scale; row maxima over the quad that shares a row
    float mx_a = -INFINITY, mx_b = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int col = 8 * nt + 2 * tig + c, j = j0 + col;
        sc[nt][c] = vis[col] && j <= lim_a ? sc[nt][c] * scale : -INFINITY;
        sc[nt][2 + c] = vis[col] && j <= lim_b ? sc[nt][2 + c] * scale : -INFINITY;
        mx_a = fmaxf(mx_a, sc[nt][c]);
        mx_b = fmaxf(mx_b, sc[nt][2 + c]);
      }
#pragma unroll
    for (int o_ = 1; o_ <= 2; o_ <<= 1) {
      mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, o_));
      mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, o_));
    }
    const float mn_a = fmaxf(m_a, mx_a), mn_b = fmaxf(m_b, mx_b);
    const float al_a = m_a == -INFINITY ? 0.f : expf(m_a - mn_a), al_b = m_b == -INFINITY ? 0.f : expf(m_b - mn_b);
    float su_a = 0.f, su_b = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        sc[nt][c] = sc[nt][c] == -INFINITY ? 0.f : expf(sc[nt][c] - mn_a);
        sc[nt][2 + c] = sc[nt][2 + c] == -INFINITY ? 0.f : expf(sc[nt][2 + c] - mn_b);
        su_a += sc[nt][c];
        su_b += sc[nt][2 + c];
      }
#pragma unroll
    for (int o_ = 1; o_ <= 2; o_ <<= 1) {
      su_a += __shfl_xor_sync(0xffffffffu, su_a, o_);
      su_b += __shfl_xor_sync(0xffffffffu, su_b, o_);
    }
    l_a = l_a * al_a + su_a;
    l_b = l_b * al_b + su_b;
    m_a = mn_a;
    m_b = mn_b;
#pragma unroll
    for (int nd = 0; nd < ND; ++nd) {
      o[nd][0] *= al_a;
      o[nd][1] *= al_a;
      o[nd][2] *= al_b;
      o[nd][3] *= al_b;
    }
    // O += P V: the score accumulators of n-tiles 2 kk, 2 kk + 1 are the A
    // fragment of entries 16 kk .. + 15
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      uint32_t ph[4], pl[4];
      split_h2(sc[2 * kk][0], sc[2 * kk][1], ph[0], pl[0]);
      split_h2(sc[2 * kk][2], sc[2 * kk][3], ph[1], pl[1]);
      split_h2(sc[2 * kk + 1][0], sc[2 * kk + 1][1], ph[2], pl[2]);
      split_h2(sc[2 * kk + 1][2], sc[2 * kk + 1][3], ph[3], pl[3]);
      const int mtx = lane >> 3, er = 16 * kk + 8 * (mtx & 1) + (lane & 7);
#pragma unroll
      for (int nd = 0; nd < ND; nd += 2) {
        uint32_t v0, v1, v2, v3;
        ldsm_x4_trans(&Vs[er][8 * (nd + (mtx >> 1))], v0, v1, v2, v3);
        mma16816(o[nd], ph, v0, v1);
        mma16816(o[nd], pl, v0, v1);
        mma16816(o[nd + 1], ph, v2, v3);
        mma16816(o[nd + 1], pl, v2, v3);
      }
    }
  }
  // output rows in the o projection's order (heads are whole 32-blocks)
  auto out_row = [&](int r) { return a.attn + (size_t)(t0 + r / G) * a.attn_ld + (hk * G + r % G) * D; };
  if (gridDim.z == 1) {
    const float ia = l_a > 0.f ? 1.f / l_a : 0.f, ib = l_b > 0.f ? 1.f / l_b : 0.f;
#pragma unroll
    for (int nd = 0; nd < ND; ++nd) {
      const int dcol = 8 * nd + 2 * tig, col = (dcol & ~31) + act_pos(dcol & 31);
      if (tok_a < S)
        *reinterpret_cast<uint32_t*>(out_row(ra) + col) = (uint32_t)f2h(o[nd][0] * ia) | ((uint32_t)f2h(o[nd][1] * ia) << 16);
      if (tok_b < S)
        *reinterpret_cast<uint32_t*>(out_row(rb) + col) = (uint32_t)f2h(o[nd][2] * ib) | ((uint32_t)f2h(o[nd][3] * ib) << 16);
    }
    return;
  }
  // this part's rows: (max, sum, 2 unused, output[D])
  constexpr int kRow = D + 4;
  const int blk = blockIdx.x * a.Hkv + hk;
  float* part = a.part + (size_t)blk * gridDim.z * 64 * kRow;
  float* mine = part + (size_t)blockIdx.z * 64 * kRow;
#pragma unroll
  for (int nd = 0; nd < ND; ++nd) {
    *reinterpret_cast<float2*>(mine + ra * kRow + 4 + 8 * nd + 2 * tig) = make_float2(o[nd][0], o[nd][1]);
    *reinterpret_cast<float2*>(mine + rb * kRow + 4 + 8 * nd + 2 * tig) = make_float2(o[nd][2], o[nd][3]);
  }
  if (tig == 0) {
    *reinterpret_cast<float2*>(mine + ra * kRow) = make_float2(m_a, l_a);
    *reinterpret_cast<float2*>(mine + rb * kRow) = make_float2(m_b, l_b);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    s_last = atomicAdd(a.part_cnt + blk, 1) == (int)gridDim.z - 1;
    if (s_last) a.part_cnt[blk] = 0;  // ready for the next launch
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // each row's weight of every part, then the rows' values with several parts'
  // loads in flight
  const int parts = gridDim.z;
  float* wgt = reinterpret_cast<float*>(flash_smem);  // [parts][64]
  if (tid < 64) {
    float M = -INFINITY, den = 0.f;
    for (int z = 0; z < parts; ++z) M = fmaxf(M, __ldcg(part + ((size_t)z * 64 + tid) * kRow));
    for (int z = 0; z < parts; ++z) {
      const float2 ml = __ldcg(reinterpret_cast<const float2*>(part + ((size_t)z * 64 + tid) * kRow));
      const float w = ml.x == -INFINITY ? 0.f : expf(ml.x - M);
      wgt[z * 64 + tid] = w;
      den = fmaf(ml.y, w, den);
    }
    wgt[parts * 64 + tid] = den > 0.f ? 1.f / den : 0.f;
  }
  __syncthreads();
  constexpr int kAt = 4, kRows = 128 / (D / 4);  // rows per thread and batch; rows per pass of the CTA
  const int c = 4 * (tid % (D / 4));
  for (int r0 = tid / (D / 4); r0 < 64; r0 += kAt * kRows) {
    float4 num[kAt];
#pragma unroll
    for (int i = 0; i < kAt; ++i) num[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int z = 0; z < parts; ++z)
#pragma unroll
      for (int i = 0; i < kAt; ++i) {
        const int r = r0 + i * kRows;
        const float4 v = __ldcg(reinterpret_cast<const float4*>(part + ((size_t)z * 64 + r) * kRow + 4 + c));
        const float w = wgt[z * 64 + r];
        num[i].x = fmaf(v.x, w, num[i].x);
        num[i].y = fmaf(v.y, w, num[i].y);
        num[i].z = fmaf(v.z, w, num[i].z);
        num[i].w = fmaf(v.w, w, num[i].w);
      }
#pragma unroll
    for (int i = 0; i < kAt; ++i) {
      const int r = r0 + i * kRows;
      if (t0 + r / G >= S) continue;
      const float k = wgt[parts * 64 + r];
      *reinterpret_cast<uint2*>(out_row(r) + (c & ~31) + act_pos(c & 31)) =
          make_uint2((uint32_t)f2h(num[i].x * k) | ((uint32_t)f2h(num[i].y * k) << 16),
                     (uint32_t)f2h(num[i].z * k) | ((uint32_t)f2h(num[i].w * k) << 16));
    }
  }
}

template <int D, int G>
cudaError_t launch_attn_t(const PrefillLayerArgs& a, cudaStream_t s) {
  static_assert(64 % G == 0, "64 query rows per CTA");
  constexpr int kSmem = (int)sizeof(FlashSmem<D>);
  const int blocks = (a.S + 64 / G - 1) / (64 / G), tiles = (a.P + a.S + 63) / 64;
  // parts of the cache: as many CTAs as partial slots, at least two tiles each
  // (and no more than one CTA should combine)
  const int parts = std::max(1, std::min(std::min(a.part_slots / (blocks * a.Hkv), tiles / 2), 32));
  return launch_behind(prefill_flash_kernel<D, G>, dim3(blocks, a.Hkv, parts), 128, kSmem, s, a);
}


template <int D, int G>
cudaError_t setup_attn_t() {
  return cudaFuncSetAttribute(prefill_flash_kernel<D, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(FlashSmem<D>));
}
template <int D>
cudaError_t setup_attn_d() {
  cudaError_t e = setup_attn_t<D, 1>();
  if (e == cudaSuccess) e = setup_attn_t<D, 2>();
  if (e == cudaSuccess) e = setup_attn_t<D, 4>();
  if (e == cudaSuccess) e = setup_attn_t<D, 8>();
  return e == cudaSuccess ? setup_attn_t<D, 16>() : e;
}

}  // namespace

cudaError_t launch_prefill_check(const int* token_ids, int vocab, const int* pos, int max_position, const uint8_t* mask,
                                 int P, int S, int* status, cudaStream_t s) {
  prefill_check_kernel<<<(S + 255) / 256, 256, 0, s>>>(token_ids, vocab, pos, max_position, mask, P, S, status);
  return cudaGetLastError();
}

cudaError_t launch_set_int(int* p, int v, cudaStream_t s) {
  set_int_kernel<<<1, 1, 0, s>>>(p, v);
  return cudaGetLastError();
}

cudaError_t launch_prefill_norm(const PrefillNormArgs& a, cudaStream_t s) {
  return launch_behind(prefill_norm_kernel, a.S, kNormThreads, 0, s, a);
}

cudaError_t launch_prefill_rope_append(const PrefillLayerArgs& a, cudaStream_t s) {
  const int n = a.S * ((a.Hq + a.Hkv) * (a.d / 8) + a.Hkv * a.d / 4);
  return launch_behind(prefill_rope_append_kernel, (n + 255) / 256, 256, 0, s, a);
}

cudaError_t launch_act_order(const uint16_t* x, int x_ld, int S, int Kp, uint16_t* out, int out_ld, cudaStream_t s) {
  act_order_kernel<<<(int)std::min<size_t>(((size_t)S * Kp / 4 + 255) / 256, 4096), 256, 0, s>>>(x, x_ld, S, Kp, out,
                                                                                                out_ld);
  return cudaGetLastError();
}

cudaError_t prefill_setup(int head_dim) { return head_dim == 128 ? setup_attn_d<128>() : setup_attn_d<64>(); }
size_t prefill_part_floats(int slots, int d) { return (size_t)slots * 64 * (d + 4); }

cudaError_t launch_prefill_attention(const PrefillLayerArgs& a, cudaStream_t s) {
  const int G = a.Hq / a.Hkv;
#define A(D)                                              \
  switch (G) {                                            \
    case 1: return launch_attn_t<D, 1>(a, s);             \
    case 2: return launch_attn_t<D, 2>(a, s);             \
    case 4: return launch_attn_t<D, 4>(a, s);             \
    case 8: return launch_attn_t<D, 8>(a, s);             \
    case 16: return launch_attn_t<D, 16>(a, s);           \
    default: return cudaErrorInvalidValue;                \
  }
  if (a.d == 128) { A(128) }
  if (a.d == 64) { A(64) }
#undef A
  return cudaErrorInvalidValue;
}

}  // namespace shard
