// Offline calibration of the equalization vector (Sec. 3.3): RoPE with positional interpolation
// (Eq. 12: the position index is multiplied by s inside the rotation, so a short calibration text
// sweeps the angles of a text s times longer) applied to pre-RoPE Keys, then the per-channel
// absolute maximum over all tokens and sequences of a KV head, lambda_i = max(amax_i, floor)^alpha
// (Eq. 10).  One pass over the Keys; the maxima meet in the output buffer through atomicMax on the
// bit patterns of non-negative floats, so the kernel needs no workspace.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels_attn.cuh"
#include "kernels_cache.cuh"
#include "layout.cuh"

namespace pmkvq {

// Rotation frequencies theta^(-2 pair / 128) in fp64, computed on the host once per call.
struct RopeFreqs { double f[64]; };

// max(m, |y|, |z|) where a NaN wins: its bit pattern is the largest, so the channel's maximum ends as NaN, which Eq. 10 reads as
// the floor.  Two values at a time: as max(m, |y|) one by one the kernel takes 1.4 % longer.
__device__ __forceinline__ float max_abs_or_nan(float m, float y, float z) {
  float r;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;\n" : "=f"(r) : "f"(m), "f"(y), "f"(z));
  return r;
}

// amax_bits [kv_heads][128] must be zero before the launch.  The Keys are read once, and that is what bounds the kernel
// (see launch_absmax for the measurement).  Grid: chunks of tokens x chunks of sequences.  A CTA first makes the
// (cos, sin) table of its tokens (fp64 angles, one per thread at a time); then two warps take a token.  Eight lanes share
// a vector, every lane eight channels i .. i + 7 and their rotation partners i + 64 .. (two 16-byte loads), so a lane's cos
// and sin stay in registers for a whole token and its running maxima, for one fixed KV head, for the whole CTA;
// they meet in shared memory once at the end.
constexpr int kAbsmaxThreads = 256;
constexpr int kAbsmaxTokens = 4;      // tokens in flight per CTA: two warps each
constexpr int kAbsmaxMaxTokens = 16;  // tokens of a CTA
constexpr int kAbsmaxPrefetch = 32768;  // bytes per token asked for (to L2) while the CTA makes its table: 118 -> 108 us, 64 KB 127
__global__ void __launch_bounds__(kAbsmaxThreads, 3) calib_absmax_kernel(const uint16_t *__restrict__ K, unsigned *amax_bits,
                                                                         int n_tokens, int n_seq, int kv_heads,
                                                                         int tokens_per_cta, int seqs_per_cta,
                                                                         double pos_scale, const RopeFreqs freqs) {
  __shared__ __align__(16) float2 s_cs[kAbsmaxMaxTokens][64];
  __shared__ unsigned s_max[8][kHeadDim];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t0 = blockIdx.x * tokens_per_cta, t1 = min(n_tokens, t0 + tokens_per_cta);
  const int s0 = blockIdx.y * seqs_per_cta, s1 = min(n_seq, s0 + seqs_per_cta);
  const bool aligned = (reinterpret_cast<uintptr_t>(K) & 15) == 0;
  pdl_launch_next();
  pdl_wait();
  if (tid < t1 - t0 && aligned) {
    const size_t row = (size_t)kv_heads * kHeadDim * sizeof(uint16_t);
    const uint32_t bytes = (uint32_t)min((size_t)kAbsmaxPrefetch, (size_t)(s1 - s0) * row);
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(reinterpret_cast<const uint8_t *>(K) + ((size_t)(t0 + tid) * n_seq + s0) * row),
                 "r"(bytes)
                 : "memory");
  }
  for (int i = tid; i < (t1 - t0) * 64; i += kAbsmaxThreads) {
    double sn, cs;
    sincos((double)(t0 + (i >> 6)) * pos_scale * freqs.f[i & 63], &sn, &cs);
    s_cs[i >> 6][i & 63] = make_float2((float)cs, (float)sn);
  }
  const int slot = (warp & 1) * 4 + (lane >> 3);  // vector slot of this quarter warp, 0 .. 7
  const int c0 = (lane & 7) * 8;                  // its lane's channels c0 .. c0 + 7 and c0 + 64 ..
  for (int h0 = 0; h0 < kv_heads; h0 += 8) {
    // the eight slots are dealt out over this group's heads: slot -> (head, first sequence)
    const int nh = min(8, kv_heads - h0), reps = 8 / nh, head = slot % nh;
    for (int i = tid; i < 8 * kHeadDim; i += kAbsmaxThreads) (&s_max[0][0])[i] = 0u;
    __syncthreads();
    float2 m1[4], m2[4];  // maxima of channels c0 + 2 j, + 1 and of their partners
#pragma unroll
    for (int j = 0; j < 4; ++j) m1[j] = m2[j] = make_float2(0.f, 0.f);
    if (slot < reps * nh) {
      for (int t = t0 + (warp >> 1); t < t1; t += kAbsmaxTokens) {
        float2 cs[4], sn[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 v = *reinterpret_cast<const float4 *>(&s_cs[t - t0][c0 + 2 * j]);
          cs[j] = make_float2(v.x, v.z);
          sn[j] = make_float2(v.y, v.w);
        }
        const uint16_t *src = K + (((size_t)t * n_seq + s0 + slot / nh) * kv_heads + h0 + head) * kHeadDim + c0;
        const size_t step = (size_t)reps * kv_heads * kHeadDim;
        // two vectors, a and b their channels c0 .. and the partners
        auto rotate = [&](const uint4 (&a4)[2], const uint4 (&b4)[2]) {
          const uint32_t a[2][4] = {{a4[0].x, a4[0].y, a4[0].z, a4[0].w}, {a4[1].x, a4[1].y, a4[1].z, a4[1].w}};
          const uint32_t b[2][4] = {{b4[0].x, b4[0].y, b4[0].z, b4[0].w}, {b4[1].x, b4[1].y, b4[1].z, b4[1].w}};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float2 y1[2], y2[2];
#pragma unroll
            for (int v = 0; v < 2; ++v) {
              const float2 x1 = make_float2(__uint_as_float(a[v][j] << 16), __uint_as_float(a[v][j] & 0xFFFF0000u));
              const float2 x2 = make_float2(__uint_as_float(b[v][j] << 16), __uint_as_float(b[v][j] & 0xFFFF0000u));
              // Eq. 11 with the scaled position; the sums one by one, since a packed sum of packed products comes out as a fused
              // multiply-add, which is another number than the sum of two rounded products
              const float2 c1 = __fmul2_rn(x1, cs[j]), s2 = __fmul2_rn(x2, sn[j]), s1 = __fmul2_rn(x1, sn[j]), c2 = __fmul2_rn(x2, cs[j]);
              y1[v] = make_float2(__fsub_rn(c1.x, s2.x), __fsub_rn(c1.y, s2.y));
              y2[v] = make_float2(__fadd_rn(s1.x, c2.x), __fadd_rn(s1.y, c2.y));
            }
            m1[j].x = max_abs_or_nan(m1[j].x, y1[0].x, y1[1].x); m1[j].y = max_abs_or_nan(m1[j].y, y1[0].y, y1[1].y);
            m2[j].x = max_abs_or_nan(m2[j].x, y2[0].x, y2[1].x); m2[j].y = max_abs_or_nan(m2[j].y, y2[0].y, y2[1].y);
          }
        };
        int s = s0 + slot / nh;
        if (aligned) {
          for (; s + 3 * reps < s1; s += 4 * reps, src += 4 * step) {  // four vectors in flight per lane
            uint4 a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              a[u] = __ldcs(reinterpret_cast<const uint4 *>(src + u * step));
              b[u] = __ldcs(reinterpret_cast<const uint4 *>(src + u * step + 64));
            }
#pragma unroll
            for (int u = 0; u < 4; u += 2) rotate({a[u], a[u + 1]}, {b[u], b[u + 1]});
          }
        }
        for (; s < s1; s += reps, src += step) {  // the rest, or Keys at an address no 16-byte load can take
          uint32_t aw[4], bw[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            aw[j] = src[2 * j] | ((uint32_t)src[2 * j + 1] << 16);
            bw[j] = src[64 + 2 * j] | ((uint32_t)src[64 + 2 * j + 1] << 16);
          }
          const uint4 a = make_uint4(aw[0], aw[1], aw[2], aw[3]), b = make_uint4(bw[0], bw[1], bw[2], bw[3]);
          rotate({a, a}, {b, b});
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        atomicMax(&s_max[head][c0 + 2 * j], __float_as_uint(m1[j].x));
        atomicMax(&s_max[head][c0 + 2 * j + 1], __float_as_uint(m1[j].y));
        atomicMax(&s_max[head][c0 + 2 * j + 64], __float_as_uint(m2[j].x));
        atomicMax(&s_max[head][c0 + 2 * j + 65], __float_as_uint(m2[j].y));
      }
    }
    __syncthreads();
    for (int i = tid; i < nh * kHeadDim; i += kAbsmaxThreads) {
      unsigned *dst = amax_bits + (size_t)h0 * kHeadDim + i;
      const unsigned v = (&s_max[0][0])[i];
      if (v > __ldcg(dst)) atomicMax(dst, v);  // most CTAs find a larger maximum there already
    }
    __syncthreads();
  }
}

// In place: bit pattern of amax -> lambda = max(amax, floor)^alpha (Eq. 10).
__global__ void calib_finish_kernel(float *lambda, int n, float floor_value, float alpha) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) lambda[i] = powf(fmaxf(lambda[i], floor_value), alpha);
}

// ---------------------------------------------------------------------------------------------
// alpha of Eq. 10 by grid search (Sec. 4.1.1): for every alpha of the grid, the squared error between the
// causal self-attention of the calibration tensors and the same operator on what the cache would hold
// at `bits` (Eq. 9: Queries times Lambda, Keys times Lambda^-1 quantized at 16 bit and taken down the
// Eq. 3 chain; Values quantized likewise).  Keys and Queries are rotated on the fly with the
// interpolated RoPE of Eq. 12 from a (cos, sin) table.
// ---------------------------------------------------------------------------------------------

// cos and sin of pos_scale * t * theta^(-2 pair / 128), rounded from fp64, two pairs to an entry: (cos of the even pair, cos of the odd
// one, sin of the even pair, sin of the odd one), so that packed fp32 instructions find adjacent channels in adjacent
// registers.  Entry e (pairs 2 e, 2 e + 1) of a token sits at angle_slot(e): the attention kernel's lanes take groups of eight
// pairs, lane after lane, and read the same entry of their groups at a time.
__host__ __device__ constexpr int angle_slot(int e) { return (e & 3) * 8 + (e >> 2); }
__global__ void rope_table_kernel(float *table, int n_tokens, double pos_scale, double theta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_tokens * 64) return;
  const int t = i >> 6, pair = i & 63;
  double s, c;
  sincos((double)t * pos_scale * pow(theta, -2.0 * pair / (double)kHeadDim), &s, &c);
  pdl_wait();  // the angles are made while the abs-max in front of this launch runs
  float *at = table + (size_t)t * 128 + angle_slot(pair >> 1) * 4 + (pair & 1);
  at[0] = (float)c;
  at[2] = (float)s;
}

constexpr int kMaxAlphas = 64;
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// x = hi + lo with both parts fp16: 22 significant bits (an absolute 2^-25 below 1/8), which three tensor-core
// products hi*hi + lo*hi + hi*lo carry into the fp32 accumulator.
__device__ __forceinline__ void split_half2(float x, float y, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 back = __half22float2(h), rest = __fadd2_rn(make_float2(x, y), make_float2(-back.x, -back.y));
  const __half2 l = __floats2half2_rn(rest.x, rest.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

// One token's 4 channels per lane (channels 4 lane .. 4 lane + 3): rotate by the token's angles.  The
// partner channel (+-64) sits in lane ^ 16.
__device__ __forceinline__ void rotate_token(float (&x)[4], const float4 *__restrict__ table_t, int lane) {
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    const float4 cs = table_t[angle_slot((lane & 15) * 2 + (e >> 1))];
    const float o0 = __shfl_xor_sync(0xffffffffu, x[e], 16), o1 = __shfl_xor_sync(0xffffffffu, x[e + 1], 16);
    // lanes 0..15 hold x1 (channel < 64): y1 = x1 c - x2 s;  lanes 16..31 hold x2: y2 = x1 s + x2 c
    x[e] = lane < 16 ? __fsub_rn(__fmul_rn(x[e], cs.x), __fmul_rn(o0, cs.z)) : __fadd_rn(__fmul_rn(o0, cs.z), __fmul_rn(x[e], cs.x));
    x[e + 1] = lane < 16 ? __fsub_rn(__fmul_rn(x[e + 1], cs.y), __fmul_rn(o1, cs.w)) : __fadd_rn(__fmul_rn(o1, cs.w), __fmul_rn(x[e + 1], cs.y));
  }
}

// Eq. 1-2 at 16 bit on one token's 128 channels spread over a warp and the Eq. 3 chain to `bits`: x becomes the code minus
// half the largest code (exact in fp32, and in one fp16 up to 8 bit), so that the dequantized value is scale * x + zero
// with the middle of the token's range as `zero`.
__device__ __forceinline__ void quantize_token_centred(float (&x)[4], int bits, float &scale, float &zero) {
  float mn = fminf(fminf(x[0], x[1]), fminf(x[2], x[3]));
  float mx = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  const float s16 = __fdiv_rn(__fsub_rn(mx, mn), 65535.0f);
  const bool plain = s16 >= 0x1p-60f && s16 <= 0x1p60f;  // else: constant token (0 / 0 converts to code 0) or absurd range
  const float y = plain ? __frcp_rn(s16) : 0.f;
  const float half = 0.5f * (float)((1 << bits) - 1);
  // the chain as one fused multiply-add (see chain_code; 1 / 1 at 16 bit), everything in whole floats
  const float inv = bits == 2 ? inv_chain_divisor<2>() : bits == 4 ? inv_chain_divisor<4>() : bits == 8 ? inv_chain_divisor<8>() : 1.0f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float d = __fsub_rn(x[e], mn);
    const float c16 = plain ? __fadd_rn(__fadd_rn(quotient_rn(d, s16, y), 8388608.0f), -8388608.0f)
                            : (float)min(max(__float2int_rn(__fdiv_rn(d, s16)), 0), 65535);
    x[e] = __fadd_rn(__fadd_rn(__fmaf_rn(c16, inv, 8388608.0f), -8388608.0f), -half);
  }
  scale = chain_scale(s16, bits);
  zero = fmaf(scale, half, mn);
}

__device__ __forceinline__ void load_bf16x4(const uint16_t *src, bool aligned, float (&x)[4]) {
  uint2 raw;
  if (aligned) raw = *reinterpret_cast<const uint2 *>(src);
  else raw = make_uint2(src[0] | ((uint32_t)src[1] << 16), src[2] | ((uint32_t)src[3] << 16));  // a caller's tensor may sit at any bf16 address
  x[0] = __uint_as_float(raw.x << 16);
  x[1] = __uint_as_float(raw.x & 0xFFFF0000u);
  x[2] = __uint_as_float(raw.y << 16);
  x[3] = __uint_as_float(raw.y & 0xFFFF0000u);
}

// ---- tensors of a pass as the attention kernel reads them ----------------------------------------------------
// Slice s = (sequence, KV head), s = seq * kv_heads + head, is cut into tiles of 64 tokens (the last one shorter).  A tile of
// r tokens is PLANES planes of r * 256 bytes, each [16 groups of 8 channels][r tokens][8 channels] fp16: one bulk copy (or one
// per channel group, for the short tile) puts it into shared memory in the core-matrix order of the MMAs, as the K-major
// operand of the scores and as the MN-major operand of the outputs alike.  One plane holds centred codes, two planes hold
// fp16 hi and lo parts of a value.  Per token a scale and a zero-point (not for plain values): [slice][n4] fp32 each, n4 = tokens
// rounded up to 4, the padding zero.
constexpr int kGridTile = 64;
constexpr int kGridMaxBatch = 4;  // alphas whose Keys sit in the workspace side by side (codes up to 8 bit)
__host__ __device__ constexpr int grid_n4(int n_tokens) { return (n_tokens + 3) & ~3; }

struct GridPrep {
  const float *amax;       // [kv_heads][128]
  const float4 *table;     // [n_tokens][32]
  const uint16_t *k, *v;   // bf16 [n_tokens][n_seq][kv_heads][128]
  int n_keys;              // outputs 0 .. n_keys - 1 are Keys (rotated and, quantized, equalized), one per alpha; the one behind them Values
  float alphas[kGridMaxBatch];
  uint8_t *out[kGridMaxBatch + 1];
  float *scale[kGridMaxBatch + 1], *zero[kGridMaxBatch + 1];
  unsigned *vmax;          // per slice, the largest scale of the Values
  int quantize;            // or keep plain
  int n_tokens, n_seq, kv_heads, bits;
  float floor_value;
};
// One CTA per (slice, tile) and output, a warp on eight vectors; they leave through shared memory as whole 16-byte pieces.  (One
// CTA for the four alphas of a batch reads its Keys once, but the latency of four rounds showed: 38 us per batch of
// 2048 x 2 x 4 vectors.)
constexpr int kPrepChunkStride = kGridTile * 16 + 16;  // padded: the 16 channel groups a warp writes fall into different banks
template <int PLANES>
__global__ void __launch_bounds__(256) alpha_grid_prep_kernel(const __grid_constant__ GridPrep p) {
  __shared__ __align__(16) uint8_t s_tile[PLANES][16 * kPrepChunkStride];
  __shared__ float s_scale[kGridTile], s_zero[kGridTile];
  __shared__ __align__(16) float s_inv[kHeadDim];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_tiles = (p.n_tokens + kGridTile - 1) / kGridTile;
  const int tile = (int)(blockIdx.x % (unsigned)n_tiles), slice = (int)(blockIdx.x / (unsigned)n_tiles), n_slices = p.n_seq * p.kv_heads;
  const int t0 = tile * kGridTile, rows = min(kGridTile, p.n_tokens - t0), n4 = grid_n4(p.n_tokens);
  const int a = blockIdx.y;
  const bool is_key = a < p.n_keys;
  const uint16_t *src = is_key ? p.k : p.v;
  const bool aligned = (reinterpret_cast<uintptr_t>(src) & 7) == 0;
  float x0[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int t = t0 + min(warp + 8 * i, rows - 1);
    load_bf16x4(src + ((size_t)t * n_slices + slice) * kHeadDim + 4 * lane, aligned, x0[i]);
  }
  if (is_key) {
#pragma unroll
    for (int i = 0; i < 8; ++i) rotate_token(x0[i], p.table + (size_t)(t0 + min(warp + 8 * i, rows - 1)) * 32, lane);
  }
  if (is_key && p.quantize) {
    if (tid < kHeadDim)
      s_inv[tid] = __fdiv_rn(1.0f, powf(fmaxf(p.amax[(size_t)(slice % p.kv_heads) * kHeadDim + tid], p.floor_value), p.alphas[a]));
    __syncthreads();
  }
  float smax = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = warp + 8 * i;
    float (&x)[4] = x0[i];
    if (p.quantize) {
      if (is_key) {
        const float4 il = *reinterpret_cast<const float4 *>(s_inv + 4 * lane);
        x[0] = __fmul_rn(x[0], il.x); x[1] = __fmul_rn(x[1], il.y); x[2] = __fmul_rn(x[2], il.z); x[3] = __fmul_rn(x[3], il.w);
      }
      float scale, zero;
      quantize_token_centred(x, p.bits, scale, zero);
      smax = fmaxf(smax, scale);
      if (lane == 0) { s_scale[row] = row < rows ? scale : 0.f; s_zero[row] = row < rows ? zero : 0.f; }
    }
    uint2 hi, lo;
    split_half2(x[0], x[1], hi.x, lo.x);
    split_half2(x[2], x[3], hi.y, lo.y);
    const int at = (lane >> 1) * kPrepChunkStride + row * 16 + (lane & 1) * 8;
    *reinterpret_cast<uint2 *>(&s_tile[0][at]) = hi;
    if constexpr (PLANES == 2) *reinterpret_cast<uint2 *>(&s_tile[1][at]) = lo;
  }
  if (!is_key && p.quantize && lane == 0) atomicMax(p.vmax + slice, __float_as_uint(smax));  // scale >= 0: uint order = float order
  __syncthreads();
  uint8_t *dst = p.out[a] + ((size_t)slice * p.n_tokens + t0) * (size_t)(256 * PLANES);
#pragma unroll
  for (int pl = 0; pl < PLANES; ++pl)
    for (int i = tid; i < 16 * rows; i += 256) {
      const int g = i / rows, r = i - g * rows;
      *reinterpret_cast<uint4 *>(dst + ((size_t)pl * 16 * rows + i) * 16) = *reinterpret_cast<const uint4 *>(&s_tile[pl][g * kPrepChunkStride + r * 16]);
    }
  if (p.quantize && tid < grid_n4(rows)) {
    p.scale[a][(size_t)slice * n4 + t0 + tid] = s_scale[tid];
    p.zero[a][(size_t)slice * n4 + t0 + tid] = s_zero[tid];
  }
}

// ---- causal self-attention of the passes ------------------------------------------------------------------------
// Grid: (sequences x query heads, alphas of the batch, query blocks from the longest to the shortest); a CTA takes 256
// queries, two tiles of 128, against their Keys in tiles of 64.  With at most 128 tokens (one tile) the two tiles are two query heads of
// one KV head instead, and the grid has a CTA per pair: a CTA of a short sequence is a chain of 10 us, whatever its second half does
// (64 tokens x 64 sequences x 8 heads,
// four alphas: 196 us a call, 264 with a CTA per head, two more launches, three more clears and one more copy to the host). Both contractions run on tcgen05.mma (fp16 in, fp32
// accumulators in tensor memory): S[query, key] = Q K^T with both operands in shared memory, O[query, channel] += P V with P
// in tensor memory, where it overwrites the scores it came from.  Warps:
//   0-3, 4-7   one warpgroup per query tile, thread = query: builds the tile's Q operand (rotated, equalized, scaled by a power of
//              two, split), then per key tile reads its 64 scores, takes probabilities against a running reference that
//              only moves when a score exceeds it by more than 8 (log2 units; the thread then rescales its own row of O),
//              and writes the weights back;
//   8, 9       one per query tile, issue its MMAs: scores of key tile j + 1, then outputs of key tile j, so the softmax of one tile
//              runs under the MMAs of the others.  (A satisfied barrier wait costs a warp about 150 cycles and a batch of MMAs waits
//              for two or three: one warp for both tiles took 4500 cycles per key tile, the MMAs take 2600.)
//   10         the bulk copies of K, V, scales and zero-points, as far ahead as the rings have room.
// Arithmetic.  The loss is a small difference of two attention outputs, so plain fp16 operands would drown it.  Queries and weights
// are sums of two fp16 numbers (22 bits).  A quantized Key or Value is scale * code + zero per token, and the centred code
// is one exact fp16 up to 8 bit, so q . k = scale_K (q . c) + zero_K sum(q) and sum p v = sum (p scale_V) c + sum p zero_V take
// two products where values split in two (the unquantized pass, 16-bit codes) take three.  Scale and zero-point work is fp32.
constexpr int kGridThreads = 352;
constexpr int kGridQTile = 128, kGridQueries = 256;
constexpr int kGridKSlots = 2, kGridVSlots = 3, kGridMetaSlots = 4;
constexpr int kGridPlaneBytes = kGridTile * 256;   // one plane of a tile
constexpr int kGridQBytes = kGridQTile * 256;      // one part (hi or lo) of a query tile's operand
constexpr int kGridSmemQ = 0, kGridSmemK = kGridSmemQ + 4 * kGridQBytes, kGridSmemV = kGridSmemK + kGridKSlots * kGridPlaneBytes,
              kGridSmemMeta = kGridSmemV + kGridVSlots * kGridPlaneBytes, kGridMetaBytes = 4 * kGridTile * 4,
              kGridSmemBytes = kGridSmemMeta + kGridMetaSlots * kGridMetaBytes;
constexpr int kGridTmemS = 0, kGridTmemO = 256;    // scores / weights [query tile][buffer] 64 columns each, outputs 128 columns each
constexpr int kGridUnitLog2 = 6;                   // weights stay below 2^(6 + 8): fp16 with room
constexpr float kGridMaxAhead = 8.0f;

__host__ __device__ constexpr bool grid_head_pairs(int n_tokens) { return n_tokens <= kGridQTile; }
struct GridAttn {
  const uint16_t *Q;       // bf16 [n_tokens][n_seq][kv_heads * group][128] before RoPE
  const uint8_t *k[kGridMaxBatch], *v;
  const float *k_scale[kGridMaxBatch], *k_zero[kGridMaxBatch], *v_scale, *v_zero;
  const unsigned *vmax;    // per slice
  const float *amax;
  const float4 *table;
  float alphas[kGridMaxBatch];  // those of this batch
  float *o_ref;            // the unquantized outputs, [sequence x head][tile of 128 queries][32 groups of 4 channels][rows][4] fp32
  double *loss_sums;       // those of this batch
  unsigned *error_word;
  int n_tokens, n_seq, kv_heads, group;
  float floor_value;
};

struct GridShared {
  unsigned long long k_full[kGridKSlots], k_free[kGridKSlots], v_full[kGridVSlots], v_free[kGridVSlots], m_full[kGridMetaSlots];
  unsigned long long q_full[2], s_full[2][2], p_full[2][2], o_done[2][2];  // [query tile][key tile mod 2]: a parity wait is never two phases off
  uint32_t tmem_base;
  int abort;
  __align__(16) float lam[kHeadDim];
};

// One warp waits for a phase of a barrier.  False if the wait ran out, here or elsewhere in the CTA: the warp then leaves its loop
// (nothing more is copied, issued or arrived at).
__device__ __forceinline__ bool grid_wait(GridShared &sh, const unsigned long long *bar, uint32_t parity, unsigned *error_word) {
  const uint32_t addr = tc05::smem_u32(bar);
  bool ok = tc05::mbar_test_wait(addr, parity & 1u);
  if (!ok) {
    for (uint32_t i = 0; !ok && i < tc05::kWaitLimit && *reinterpret_cast<volatile int *>(&sh.abort) == 0; ++i)
      ok = tc05::mbar_try_wait_hint(addr, parity & 1u, tc05::kWaitHintNs);
    if (!ok) {
      sh.abort = 1;
      atomicOr(error_word, 1u);
    }
  }
  return __all_sync(0xffffffffu, ok);
}

// PLANES: planes of K and V.  SCALED: quantized tensors with scales and zero-points, whose outputs are compared with o_ref;
// otherwise the unquantized operator, whose outputs are kept there.
template <int PLANES, bool SCALED>
__global__ void __launch_bounds__(kGridThreads, 1) alpha_grid_attn_kernel(const __grid_constant__ GridAttn p) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ GridShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q_heads = p.kv_heads * p.group, batch = blockIdx.y;
  const bool pairs = grid_head_pairs(p.n_tokens);
  const int per_kv = pairs ? (p.group + 1) / 2 : p.group;  // CTAs of a KV head
  const int slice = (int)blockIdx.x / per_kv, in_slice = (int)blockIdx.x - slice * per_kv;
  const int seq = slice / p.kv_heads, kv_head = slice - seq * p.kv_heads;
  const int head0 = kv_head * p.group + (pairs ? 2 * in_slice : in_slice);  // query head of the first tile
  const int q_block = ((int)gridDim.z - 1 - (int)blockIdx.z) * kGridQueries;  // long rows first
  const int n = p.n_tokens, n4 = grid_n4(n);
  int nt[2];  // key tiles of the two query tiles
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int first = pairs ? 0 : q_block + q * kGridQTile;
    const bool any = pairs ? 2 * in_slice + q < p.group : first < n;
    nt[q] = any ? (min(n, first + kGridQTile) - 1) / kGridTile + 1 : 0;
  }
  const int n_kt = max(nt[0], nt[1]);
  const bool ragged = n_kt * kGridTile > n;  // the last tile is the slice's short one

  if (tid == 0) {
    const uint32_t users = nt[1] > 0 ? 2 : 1;  // query tiles whose MMAs read a slot
    for (int i = 0; i < kGridKSlots; ++i) { tc05::mbar_init(tc05::smem_u32(&sh.k_full[i]), 1); tc05::mbar_init(tc05::smem_u32(&sh.k_free[i]), users); }
    for (int i = 0; i < kGridVSlots; ++i) { tc05::mbar_init(tc05::smem_u32(&sh.v_full[i]), 1); tc05::mbar_init(tc05::smem_u32(&sh.v_free[i]), users); }
    for (int i = 0; i < kGridMetaSlots; ++i) tc05::mbar_init(tc05::smem_u32(&sh.m_full[i]), 1);
    for (int q = 0; q < 2; ++q) {
      for (int b = 0; b < 2; ++b) { tc05::mbar_init(tc05::smem_u32(&sh.s_full[q][b]), 1); tc05::mbar_init(tc05::smem_u32(&sh.p_full[q][b]), 4); }
      tc05::mbar_init(tc05::smem_u32(&sh.q_full[q]), 4);
      for (int b = 0; b < 2; ++b) tc05::mbar_init(tc05::smem_u32(&sh.o_done[q][b]), 1);
    }
    sh.abort = 0;
    tc05::mbar_init_fence();
  }
  if (warp == 8) tc05::tmem_alloc(tc05::smem_u32(&sh.tmem_base), 512);
  if (tid < kHeadDim) {  // what the rotated queries are multiplied by: lambda and the softmax scale in log2 units
    const float scale_log2 = 1.4426950408889634f * rsqrtf((float)kHeadDim);
    sh.lam[tid] = SCALED ? powf(fmaxf(p.amax[(size_t)kv_head * kHeadDim + tid], p.floor_value), p.alphas[batch]) * scale_log2 : scale_log2;
  }
  if (ragged) {  // rows behind the last token stay as they are in the operands: they must be finite
    for (int i = kGridSmemK + 16 * tid; i < kGridSmemBytes; i += 16 * kGridThreads) *reinterpret_cast<uint4 *>(smem + i) = make_uint4(0u, 0u, 0u, 0u);
    tc05::fence_async_smem();
  }
  tc05::fence_before_sync();
  __syncthreads();
  tc05::fence_after_sync();
  const uint32_t tmem = sh.tmem_base;
  const uint32_t s_base = tc05::smem_u32(smem);
  auto wait = [&](const unsigned long long *bar, int phase) { return grid_wait(sh, bar, (uint32_t)phase, p.error_word); };

  if (warp == 10) {
    // ---- copies ----
    const uint8_t *k_src = p.k[batch] + (size_t)slice * n * (256 * PLANES), *v_src = p.v + (size_t)slice * n * (256 * PLANES);
    auto tile_copy = [&](uint32_t dst, const uint8_t *src, int rows, const unsigned long long *bar) {
      if (lane == 0) {
        const uint32_t b = tc05::smem_u32(bar);
        tc05::mbar_arrive_expect_tx(b, (uint32_t)rows * 256u);
        if (rows == kGridTile) {
          tc05::bulk_g2s(dst, src, kGridPlaneBytes, b);
        } else {
          for (int g = 0; g < 16; ++g) tc05::bulk_g2s(dst + g * (kGridTile * 16), src + (size_t)g * rows * 16, (uint32_t)rows * 16u, b);
        }
      }
      __syncwarp();
    };
    bool go = true;
    for (int j = 0; go && j < n_kt; ++j) {
      const int rows = min(kGridTile, n - j * kGridTile);
      for (int pl = 0; pl < PLANES; ++pl) {
        const int a = j * PLANES + pl, slot = a % kGridKSlots;
        if (!go || (a >= kGridKSlots && !(go = wait(&sh.k_free[slot], a / kGridKSlots - 1)))) break;
        tile_copy(s_base + kGridSmemK + slot * kGridPlaneBytes, k_src + ((size_t)j * kGridTile * PLANES + (size_t)pl * rows) * 256, rows, &sh.k_full[slot]);
      }
      if constexpr (SCALED) {
        // slot j mod 4 was last read for tile j - 4, whose weights were all written before the scores of tile j - 2 that freed
        // this tile's K slot could be issued (a query tile without a tile j - 2 has no tile j - 4 to be read late either)
        if (lane == 0 && go) {
          const uint32_t b = tc05::smem_u32(&sh.m_full[j % kGridMetaSlots]), bytes = (uint32_t)grid_n4(rows) * 4u;
          const uint32_t dst = s_base + kGridSmemMeta + (j % kGridMetaSlots) * kGridMetaBytes;
          const size_t at = (size_t)slice * n4 + (size_t)j * kGridTile;
          tc05::mbar_arrive_expect_tx(b, 4u * bytes);
          tc05::bulk_g2s(dst, p.k_scale[batch] + at, bytes, b);
          tc05::bulk_g2s(dst + kGridTile * 4, p.k_zero[batch] + at, bytes, b);
          tc05::bulk_g2s(dst + 2 * kGridTile * 4, p.v_scale + at, bytes, b);
          tc05::bulk_g2s(dst + 3 * kGridTile * 4, p.v_zero + at, bytes, b);
        }
        __syncwarp();
      }
      for (int pl = 0; pl < PLANES; ++pl) {
        const int a = j * PLANES + pl, slot = a % kGridVSlots;
        if (!go || (a >= kGridVSlots && !(go = wait(&sh.v_free[slot], a / kGridVSlots - 1)))) break;
        tile_copy(s_base + kGridSmemV + slot * kGridPlaneBytes, v_src + ((size_t)j * kGridTile * PLANES + (size_t)pl * rows) * 256, rows, &sh.v_full[slot]);
      }
    }
  } else if (warp >= 8) {
    // ---- MMAs of query tile q ----
    const int q = warp - 8, n_mine = nt[q];
    constexpr uint32_t idesc_s = tc05::idesc_f16(128, kGridTile, 0), idesc_o = tc05::idesc_f16(128, kHeadDim, 1);
    const uint64_t qh = tc05::smem_desc(s_base + kGridSmemQ + 2 * q * kGridQBytes, kGridQTile * 16, 128);
    const uint64_t ql = tc05::smem_desc(s_base + kGridSmemQ + (2 * q + 1) * kGridQBytes, kGridQTile * 16, 128);
    bool go = true;
    auto scores = [&](int j) {
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) go = go && wait(&sh.k_full[(j * PLANES + pl) % kGridKSlots], (j * PLANES + pl) / kGridKSlots);
      // the output MMAs that read this buffer's weights are complete; the query operand is there
      go = go && (j >= 2 ? wait(&sh.o_done[q][j & 1], (j >> 1) - 1) : j == 0 ? wait(&sh.q_full[q], 0) : true);
      if (!go) return;
      tc05::fence_after_sync();
      const uint32_t d = tmem + kGridTmemS + 64 * (2 * q + (j & 1));
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) {
        const uint64_t kd = tc05::smem_desc(s_base + kGridSmemK + ((j * PLANES + pl) % kGridKSlots) * kGridPlaneBytes, kGridTile * 16, 128);
        // 16 channels per MMA: two channel groups
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) tc05::mma_f16_ss_elect(d, qh + ks * (2 * kGridQTile), kd + ks * (2 * kGridTile), idesc_s, pl > 0 || ks > 0 ? 1u : 0u);
        if (pl == 0) {
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) tc05::mma_f16_ss_elect(d, ql + ks * (2 * kGridQTile), kd + ks * (2 * kGridTile), idesc_s, 1u);
        }
      }
      tc05::mma_commit_elect(tc05::smem_u32(&sh.s_full[q][j & 1]));
      // a slot is given back only if a later tile will use it: no arrival may be on its way when the CTA ends
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) {
        const int a = j * PLANES + pl;
        if (a + kGridKSlots < n_kt * PLANES) tc05::mma_commit_elect(tc05::smem_u32(&sh.k_free[a % kGridKSlots]));
      }
    };
    auto outputs = [&](int j) {
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) go = go && wait(&sh.v_full[(j * PLANES + pl) % kGridVSlots], (j * PLANES + pl) / kGridVSlots);
      go = go && wait(&sh.p_full[q][j & 1], j >> 1);
      if (!go) return;
      tc05::fence_after_sync();
      const uint32_t d = tmem + kGridTmemO + 128 * q, w_hi = tmem + kGridTmemS + 64 * (2 * q + (j & 1)), w_lo = w_hi + 32;
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) {
        const uint64_t vd = tc05::smem_desc(s_base + kGridSmemV + ((j * PLANES + pl) % kGridVSlots) * kGridPlaneBytes, 128, kGridTile * 16);
        // 16 keys per MMA: two rows of core matrices
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) tc05::mma_f16_ts_elect(d, w_hi + 8 * ks, vd + ks * 16, idesc_o, j > 0 || pl > 0 || ks > 0 ? 1u : 0u);
        if (pl == 0) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) tc05::mma_f16_ts_elect(d, w_lo + 8 * ks, vd + ks * 16, idesc_o, 1u);
        }
      }
      tc05::mma_commit_elect(tc05::smem_u32(&sh.o_done[q][j & 1]));
#pragma unroll
      for (int pl = 0; pl < PLANES; ++pl) {
        const int a = j * PLANES + pl;
        if (a + kGridVSlots < n_kt * PLANES) tc05::mma_commit_elect(tc05::smem_u32(&sh.v_free[a % kGridVSlots]));
      }
    };
    if (n_mine > 0) scores(0);
    for (int j = 0; go && j < n_mine; ++j) {
      if (j + 1 < n_mine) scores(j + 1);
      if (go) outputs(j);
    }
    // The key tiles that only the second query tile uses: nothing of this warp reads them.  It gives a slot back once the tile is
    // there (the slot's earlier uses are then all over, so no arrival is counted for the wrong use).
    for (int a = n_mine * PLANES; go && n_mine > 0 && a < n_kt * PLANES; ++a) {
      if (a + kGridKSlots < n_kt * PLANES) {
        go = go && wait(&sh.k_full[a % kGridKSlots], a / kGridKSlots);
        if (lane == 0 && go) tc05::mbar_arrive(tc05::smem_u32(&sh.k_free[a % kGridKSlots]));
      }
      if (a + kGridVSlots < n_kt * PLANES) {
        go = go && wait(&sh.v_full[a % kGridVSlots], a / kGridVSlots);
        if (lane == 0 && go) tc05::mbar_arrive(tc05::smem_u32(&sh.v_free[a % kGridVSlots]));
      }
      __syncwarp();
    }
  } else if (nt[warp >> 2] > 0) {
    // ---- a query tile ----
    const int q = warp >> 2, row = tid & 127;
    const int first_q = pairs ? 0 : q_block + q * kGridQTile, q_head = head0 + (pairs ? q : 0);
    const int qi = min(first_q + row, n - 1);  // a dead row repeats the last query; its output is dropped
    const bool alive = first_q + row < n;
    const uint32_t t_lane = (uint32_t)((warp & 3) * 32) << 16;
    float sum_q = 0.f, f = 1.f;  // sum of the operand's elements; scores are f times the dot products
    {
      // Eight rows at a time, four lanes on a row, each with the channels of two groups and of their partner groups (+ 8).  Loads then
      // take whole 64-byte pieces (thread = row would touch 32 lines per load and took 60 000 cycles), and the eight lanes
      // of a store phase write eight consecutive rows of the operand (eight lanes on a row write groups 2 KB apart, a bank
      // conflict of eight).  The loop is not unrolled: straight-line code that a CTA runs once costs more to fetch than to run.
      const bool aligned = (reinterpret_cast<uintptr_t>(p.Q) & 15) == 0;
#pragma unroll 1
      for (int rg = 0; rg < 4; ++rg) {
        const int r = (warp & 3) * 32 + 8 * rg + (lane & 7), t = min(first_q + r, n - 1);
        const uint16_t *src = p.Q + (((size_t)t * p.n_seq + seq) * q_heads + q_head) * kHeadDim + 8 * (lane >> 3);
        const float4 *tab = p.table + (size_t)t * 32 + (lane >> 3);
        uint4 raw[2][2];  // [half of the groups][channels, partners]
        float4 cs[2][4];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          if (aligned) {
            raw[g][0] = __ldg(reinterpret_cast<const uint4 *>(src + 32 * g));
            raw[g][1] = __ldg(reinterpret_cast<const uint4 *>(src + 32 * g + 64));
          } else {
            uint32_t w[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const uint16_t *at = src + 32 * g + 2 * (c & 3) + 64 * (c >> 2);
              w[c] = at[0] | ((uint32_t)at[1] << 16);
            }
            raw[g][0] = make_uint4(w[0], w[1], w[2], w[3]);
            raw[g][1] = make_uint4(w[4], w[5], w[6], w[7]);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) cs[g][c] = __ldg(tab + 4 * g + 8 * c);  // entries 4 group + c
        }
        float2 y1[2][4], y2[2][4];
        float mx = 0.f;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int ch = 8 * (4 * g + (lane >> 3));
          const uint32_t r1[4] = {raw[g][0].x, raw[g][0].y, raw[g][0].z, raw[g][0].w}, r2[4] = {raw[g][1].x, raw[g][1].y, raw[g][1].z, raw[g][1].w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {  // channels 2 c, 2 c + 1 of the group and their partners
            const float2 co = make_float2(cs[g][c].x, cs[g][c].y), si = make_float2(cs[g][c].z, cs[g][c].w);
            const float2 x1 = make_float2(__uint_as_float(r1[c] << 16), __uint_as_float(r1[c] & 0xFFFF0000u));
            const float2 x2 = make_float2(__uint_as_float(r2[c] << 16), __uint_as_float(r2[c] & 0xFFFF0000u));
            const float2 l1 = *reinterpret_cast<const float2 *>(&sh.lam[ch + 2 * c]), l2 = *reinterpret_cast<const float2 *>(&sh.lam[ch + 2 * c + 64]);
            y1[g][c] = __fmul2_rn(__ffma2_rn(__fmul2_rn(x2, si), make_float2(-1.f, -1.f), __fmul2_rn(x1, co)), l1);
            y2[g][c] = __fmul2_rn(__fadd2_rn(__fmul2_rn(x1, si), __fmul2_rn(x2, co)), l2);
            mx = fmaxf(fmaxf(mx, fmaxf(fabsf(y1[g][c].x), fabsf(y1[g][c].y))), fmaxf(fabsf(y2[g][c].x), fabsf(y2[g][c].y)));
          }
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
        const int shift = mx > 0.f ? max(-100, min(100, 136 - (int)(__float_as_uint(mx) >> 23))) : 0;  // largest element to [2^9, 2^10)
        const float2 up = make_float2(exp2i(shift), exp2i(shift));
        float2 sum2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint8_t *q_op = smem + kGridSmemQ + 2 * q * kGridQBytes + (4 * g + (lane >> 3)) * (kGridQTile * 16) + r * 16;
          uint32_t h1[4], o1[4], h2[4], o2[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float2 a = __fmul2_rn(y1[g][c], up), b = __fmul2_rn(y2[g][c], up);
            sum2 = __fadd2_rn(sum2, __fadd2_rn(a, b));
            split_half2(a.x, a.y, h1[c], o1[c]);
            split_half2(b.x, b.y, h2[c], o2[c]);
          }
          *reinterpret_cast<uint4 *>(q_op) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
          *reinterpret_cast<uint4 *>(q_op + kGridQBytes) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
          *reinterpret_cast<uint4 *>(q_op + 8 * (kGridQTile * 16)) = make_uint4(h2[0], h2[1], h2[2], h2[3]);
          *reinterpret_cast<uint4 *>(q_op + kGridQBytes + 8 * (kGridQTile * 16)) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
        }
        float sum = sum2.x + sum2.y;
        sum += __shfl_xor_sync(0xffffffffu, sum, 8);
        sum += __shfl_xor_sync(0xffffffffu, sum, 16);
        if ((lane >> 3) == rg) { sum_q = sum; f = exp2i(-shift); }  // row L of the warp is lane L's from here on
      }
      tc05::fence_async_smem();
      warp_arrive(&sh.q_full[q], lane);
    }
    // Probabilities are taken times 2^bias: with the weights' unit folded in, numerator and denominator share the factor.
    float bias = (float)kGridUnitLog2;
    if constexpr (SCALED) {
      const unsigned vm = __ldg(p.vmax + slice);
      if (vm) bias -= (float)max((int)(vm >> 23) - 126, -60);
    }
    float m = -INFINITY;      // reference (below every score at first); arguments of the exponential are f * t - m_b
    float m_b = 0.f;          // m - bias
    float2 l2 = make_float2(0.f, 0.f), z2 = make_float2(0.f, 0.f);
    const uint32_t t_o = tmem + kGridTmemO + 128 * q + t_lane;
    bool go = true;
    for (int j = 0; j < nt[q]; ++j) {
      const uint32_t t_s = tmem + kGridTmemS + 64 * (2 * q + (j & 1)) + t_lane;
      const float *meta = reinterpret_cast<const float *>(smem + kGridSmemMeta + (j % kGridMetaSlots) * kGridMetaBytes);
      go = wait(&sh.s_full[q][j & 1], j >> 1);
      if constexpr (SCALED) go = go && wait(&sh.m_full[j % kGridMetaSlots], j / kGridMetaSlots);
      if (!go) break;
      tc05::fence_after_sync();
      float t[64];
      {
        uint32_t raw[64];
        tc05::tmem_ld32(t_s, raw);
        tc05::tmem_ld32(t_s + 32, raw + 32);
        tc05::wait_ld();
        const float2 sq2 = make_float2(sum_q, sum_q);
#pragma unroll
        for (int k = 0; k < 64; k += 4) {
          float2 d0 = make_float2(__uint_as_float(raw[k]), __uint_as_float(raw[k + 1]));
          float2 d1 = make_float2(__uint_as_float(raw[k + 2]), __uint_as_float(raw[k + 3]));
          if constexpr (SCALED) {
            const float4 sk = *reinterpret_cast<const float4 *>(meta + k), zk = *reinterpret_cast<const float4 *>(meta + kGridTile + k);
            d0 = __ffma2_rn(make_float2(sk.x, sk.y), d0, __fmul2_rn(make_float2(zk.x, zk.y), sq2));
            d1 = __ffma2_rn(make_float2(sk.z, sk.w), d1, __fmul2_rn(make_float2(zk.z, zk.w), sq2));
          }
          t[k] = d0.x; t[k + 1] = d0.y; t[k + 2] = d1.x; t[k + 3] = d1.y;
        }
      }
      if (j * kGridTile + kGridTile - 1 > first_q) {  // some key of the tile may lie behind some query of the tile
#pragma unroll
        for (int k = 0; k < 64; ++k)
          if (j * kGridTile + k > qi) t[k] = -INFINITY;
      }
      float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int k = 0; k < 64; k += 2) mx[(k >> 1) & 3] = fmaxf(mx[(k >> 1) & 3], fmaxf(t[k], t[k + 1]));
      const float top = f * fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
      if (__any_sync(0xffffffffu, top > m + kGridMaxAhead)) {
        // key 0 is live for every query and sits in the first tile, so m is finite from the first tile on
        const float m_new = fmaxf(m, top);
        const float corr = ex2_fast(m - m_new);  // 0 on the first tile
        m = m_new;
        m_b = m - bias;
        l2 = __fmul2_rn(l2, make_float2(corr, corr));
        z2 = __fmul2_rn(z2, make_float2(corr, corr));
        if (j > 0) {  // this thread's row of the outputs, once all output MMAs issued so far are complete
          if (!(go = wait(&sh.o_done[q][(j - 1) & 1], (j - 1) >> 1))) break;
          tc05::fence_after_sync();
#pragma unroll 1
          for (int c = 0; c < 128; c += 32) {
            uint32_t o[32];
            tc05::tmem_ld32(t_o + c, o);
            tc05::wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
            tc05::tmem_st32(t_o + c, o);
          }
        }
      }
      const float2 f2 = make_float2(f, f), nm2 = make_float2(-m_b, -m_b);
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int k = 0; k < 32; k += 4) {
          float4 sv = make_float4(0.f, 0.f, 0.f, 0.f), zv = sv;
          if constexpr (SCALED) {
            sv = *reinterpret_cast<const float4 *>(meta + 2 * kGridTile + 32 * half + k);
            zv = *reinterpret_cast<const float4 *>(meta + 3 * kGridTile + 32 * half + k);
          }
#pragma unroll
          for (int e = 0; e < 4; e += 2) {
            const float2 arg = __ffma2_rn(f2, make_float2(t[32 * half + k + e], t[32 * half + k + e + 1]), nm2);
            const float2 pr = make_float2(ex2_fast(arg.x), ex2_fast(arg.y));
            l2 = __fadd2_rn(l2, pr);
            float2 w = pr;
            if constexpr (SCALED) {
              z2 = __ffma2_rn(pr, e ? make_float2(zv.z, zv.w) : make_float2(zv.x, zv.y), z2);
              w = __fmul2_rn(pr, e ? make_float2(sv.z, sv.w) : make_float2(sv.x, sv.y));
            }
            split_half2(w.x, w.y, hi[(k + e) / 2], lo[(k + e) / 2]);
          }
        }
        tc05::tmem_st16(t_s + 16 * half, hi);
        tc05::tmem_st16(t_s + 32 + 16 * half, lo);
      }
      tc05::wait_st();
      tc05::fence_before_sync();
      warp_arrive(&sh.p_full[q][j & 1], lane);
    }
    // ---- the pass's output: keep it (the unquantized pass) or compare with the kept one ----
    const int rows = min(kGridQTile, n - first_q);
    float4 *kept = reinterpret_cast<float4 *>(p.o_ref) + (((size_t)seq * q_heads + q_head) * n + first_q) * (kHeadDim / 4) + row;
    const float inv_l = __fdiv_rn(1.0f, l2.x + l2.y), zs = z2.x + z2.y;
    float err = 0.f;
#pragma unroll 1
    for (int c0 = 0; go && c0 < 128; c0 += 64) {
      float4 ref[16];  // half of the query's kept outputs, the first half asked for before the last output MMAs are complete
      if (SCALED && alive) {
#pragma unroll
        for (int i = 0; i < 16; ++i) ref[i] = kept[(size_t)(c0 / 4 + i) * rows];
      }
      if (c0 == 0 && !(go = wait(&sh.o_done[q][(nt[q] - 1) & 1], (nt[q] - 1) >> 1))) break;
      tc05::fence_after_sync();
#pragma unroll
      for (int c = 0; c < 64; c += 32) {
        uint32_t o[32];
        tc05::tmem_ld32(t_o + c0 + c, o);
        tc05::wait_ld();
        if (alive) {
#pragma unroll
          for (int i = 0; i < 32; i += 4) {
            float4 v = make_float4((__uint_as_float(o[i]) + zs) * inv_l, (__uint_as_float(o[i + 1]) + zs) * inv_l,
                                   (__uint_as_float(o[i + 2]) + zs) * inv_l, (__uint_as_float(o[i + 3]) + zs) * inv_l);
            if constexpr (SCALED) {
              const float4 r = ref[(c + i) / 4];
              v.x -= r.x; v.y -= r.y; v.z -= r.z; v.w -= r.w;
              err = fmaf(v.x, v.x, err); err = fmaf(v.y, v.y, err); err = fmaf(v.z, v.z, err); err = fmaf(v.w, v.w, err);
            } else {
              kept[(size_t)((c0 + c + i) / 4) * rows] = v;
            }
          }
        }
      }
    }
    if constexpr (SCALED) {
      double e = (double)err;
#pragma unroll
      for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
      if (lane == 0) atomicAdd(p.loss_sums + batch, e);
    }
  }
  tc05::fence_before_sync();
  __syncthreads();
  if (*reinterpret_cast<volatile int *>(&sh.abort)) {
    // a wait gave up: copies and MMAs may still be in flight; give them about a millisecond (a bounded delay)
    const long long c0 = clock64();
    while (clock64() - c0 < 2000000ll) {}
    __syncthreads();
  }
  if (warp == 8) tc05::tmem_dealloc(tmem, 512);
}

}  // namespace pmkvq
