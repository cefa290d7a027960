#pragma once
// Stage math of decode attention on the tensor cores (bf16 caches, several
// query heads per kv head; attn_uses_mma in internal.h says which), used by
// both decode-attention kernels.
//
// On the CUDA cores (VecMath) every K and V element is widened, and multiplied once
// per query head, so launches with G = 4 or 8 were bound by instruction issue,
// not by HBM, and the short launches of G = 2 spent most of their streaming time
// on it.  Here a warp takes 16 slots at a time through mma.sync.m16n8k16 (fp32
// accumulation): the G query heads are rows of A, the slots the columns of
// S = q K^T, and the rows of P V.  (tcgen05 wants 64 or more rows of A, eight
// times the heads there are, and a round trip through TMEM per stage.)
// Measured (us, before / now): 64 sequences of 2048-4096 slots, 64/8 heads of 128:
// 726 / 131; 32 of 4096-8192, 32/8 heads of 128: 167 / 133; 8 of up to 4096, 64/8
// heads of 64: 28.4 / 22.3; a decode step of 16 layers, 16 sequences of 2048,
// 6/3 heads of 96: 185 / 173.
//
//  * Probabilities stay fp32: p is split exactly into three bf16 terms (hi,
//    mid, lo; 24 bits), and the spare rows of A carry them.  G = 2: rows 0-1
//    hi, 2-3 mid, 4-5 lo of one MMA; G = 4: rows 0-3, 4-7, 8-11.  G = 8: two
//    MMAs, (hi | mid) and (hi | lo), with the terms taken of p / 2 so that their
//    two hi sums add up to p's.  The accumulators of hi, mid and lo stay apart
//    and are summed when a piece ends; where hi's sum is not finite (infinite V)
//    it stands alone, since 0 * inf in the smaller terms is no part of the result.
//  * No ldmatrix and no swizzle: both contractions may run over their index in
//    any order.  Lane (g, t) = (lane / 4, lane % 4) reads 16 bytes of K per
//    two MMAs, and the columns of V are dealt so that one 16-byte vector of
//    each of its four slots makes the B fragments of eight column tiles
//    (two byte permutes each).
//  * Lanes that read together then read rows four or eight apart, which at d = 64
//    and 128 start on the same bank: the V tile lies in two blocks of half the
//    stage's slots, the second shifted by 64 bytes; at d = 96 (192-byte rows)
//    half of the lanes take the rows of a pair in the other order.  Either way
//    the reads are two-way conflicted, which costs less than smaller copies: V in
//    four blocks, without conflicts, took 68.0 us where this takes 58.6 (16
//    sequences of 4000-8192 slots, 32/8 heads of 96) and 135.6 for 131.2 (128).
#include "common.cuh"
#include "internal.h"

namespace wm {
namespace attn_detail {

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&t);
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

template <int HD, int G, int SLOTS>
struct MmaMath {
  using T = __nv_bfloat16;
  static_assert(G == 2 || G == 4 || G == 8, "two, four or eight query heads");
  static_assert(SLOTS % 16 == 0 && HD % 32 == 0, "16 slots and 32 columns per step");
  static constexpr int kSub = SLOTS / 4;                       // slots of a lane per stage
  static constexpr bool kFlip = HD % 64 != 0;                  // rows of two lane pairs swapped (see above)
  static constexpr int kBlocks = kFlip ? 1 : 2;                // blocks of the V tile
  static constexpr int kSkew = 32;                             // elements between blocks
  static constexpr int kPad = kAttnMmaPad / (int)sizeof(T);    // elements added to V
  // queries come straight from L2 when a piece starts: a ring of them for three
  // stages (24 KB per CTA at G = 8, d = 128) would leave one CTA per SM
  static constexpr bool kQueryRing = false;
  static_assert((kBlocks - 1) * kSkew <= kPad, "the shift fits the padding");
  static constexpr int KV = HD / 32;                           // 16-byte K vectors per lane and slot
  static constexpr int NT = HD / 8;                            // column tiles of O
  static constexpr int FULL_I = HD / 64, TAIL = HD % 64 / 32;  // 64-column blocks, a 32-column rest

  uint32_t qa[KV][4];  // query head g % G, vector t + 4 i
  float m, l;          // head g % G: running max (of the quad), sum (of this lane's slots)
  float acc[NT][4];

  __device__ __forceinline__ static int g_of(int lane) { return lane >> 2; }

  __device__ __forceinline__ void reset() {
    m = -INFINITY;
    l = 0.f;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[n][i] = 0.f;
  }
  template <bool L2>
  __device__ __forceinline__ void load_q(const T* rows, int lane) {
    const T* r = rows + (g_of(lane) % G) * HD + (lane & 3) * 8;
#pragma unroll
    for (int i = 0; i < KV; ++i) {
      const uint4* s = reinterpret_cast<const uint4*>(r + i * 32);
      const uint4 v = L2 ? __ldcg(s) : *s;
      qa[i][0] = v.x;
      qa[i][1] = v.y;
      qa[i][2] = v.z;
      qa[i][3] = v.w;
    }
  }

  // One stage.  Slot `ls` is valid if ls < valid_slots and bit ls >> log2R
  // of mask is set; FULL: every slot is.
  template <bool FULL>
  __device__ __forceinline__ void consume(const T* Ks, const T* Vs, int lane, float qscale,
                                          int valid_slots, uint64_t mask, int log2R) {
    const int g = g_of(lane), t = lane & 3;
#pragma unroll
    for (int s = 0; s < SLOTS / 16; ++s) {
      // S: column n of tile j is slot kSub (n / 2) + 4 s + 2 j + n % 2 (kFlip: with
      // the last bit flipped in columns 4-7), so that lane (g, t) holds slots kSub t +
      // 4 s + (0..3 ^ flip), all in one V block
      float c[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
        const T* kr = Ks + (kSub * (g >> 1) + 4 * s + 2 * j + ((g ^ (kFlip ? g >> 2 : 0)) & 1)) * HD + t * 8;
#pragma unroll
        for (int i = 0; i < KV; ++i) {
          const uint4 v = *reinterpret_cast<const uint4*>(kr + i * 32);
          mma_bf16_16816(c[j], qa[i][0], 0u, qa[i][1], 0u, v.x, v.y);
          mma_bf16_16816(c[j], qa[i][2], 0u, qa[i][3], 0u, v.z, v.w);
        }
      }
      const int ls = kSub * t + 4 * s, fx = kFlip ? t >> 1 : 0;
      float sc[4];
      bool ok[4];
      float mx = -INFINITY;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ok[i] = FULL || ((ls + (i ^ fx) < valid_slots) && ((mask >> ((ls + (i ^ fx)) >> log2R)) & 1ull));
        sc[i] = ok[i] ? c[i >> 1][i & 1] * qscale : -INFINITY;
        mx = fmaxf(mx, sc[i]);
      }
      mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
      if (__any_sync(0xFFFFFFFFu, mx > m)) {  // some head's max rises: rescale
        const float mnew = fmaxf(m, mx);
        const float corr = mnew == -INFINITY ? 1.f : exp2f(m - mnew);  // 0 while m is still -inf
        l *= corr;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[n][i] *= corr;
        m = mnew;
      }
      float p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        p[i] = (FULL || sc[i] != -INFINITY) ? exp2f(sc[i] - m) : 0.f;
        l += p[i];
      }
      // p as three bf16 terms; A column k of the step is slot 4 s + {0, 1} of
      // every block for k < 8, {2, 3} for k >= 8
      uint32_t a0[2], a1[2], a2[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float f = G == 8 ? 0.5f : 1.f, r = G == 8 ? 2.f : 1.f;
        const float x = f * p[2 * j], y = f * p[2 * j + 1];
        const uint32_t hi = pack_bf16(x, y);
        const float x1 = r * (x - bf16_lo(hi)), y1 = r * (y - bf16_hi(hi));
        const uint32_t mid = pack_bf16(x1, y1);
        const uint32_t lo = pack_bf16(x1 - bf16_lo(mid), y1 - bf16_hi(mid));
        a0[j] = G == 8 || g / G == 0 ? hi : g / G == 1 ? mid : lo;
        a1[j] = G == 8 ? mid : G == 4 ? lo : 0u;
        a2[j] = lo;
      }
      auto pv = [&](float (&o)[4], uint32_t b0, uint32_t b1) {
        mma_bf16_16816(o, a0[0], a1[0], a0[1], a1[1], b0, b1);
        if (G == 8) mma_bf16_16816(o, a0[0], a2[0], a0[1], a2[1], b0, b1);
      };
      const T* vr = Vs + ls * HD + (kBlocks > 1 ? (t >> 1) * kSkew : 0);
#pragma unroll
      for (int i = 0; i < FULL_I; ++i) {
        uint32_t v[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint4 x = *reinterpret_cast<const uint4*>(vr + (r ^ fx) * HD + i * 64 + g * 8);
          if (!FULL && !ok[r]) x = make_uint4(0u, 0u, 0u, 0u);
          v[r][0] = x.x;
          v[r][1] = x.y;
          v[r][2] = x.z;
          v[r][3] = x.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          pv(acc[8 * i + 2 * e], __byte_perm(v[0][e], v[1][e], 0x5410), __byte_perm(v[2][e], v[3][e], 0x5410));
          pv(acc[8 * i + 2 * e + 1], __byte_perm(v[0][e], v[1][e], 0x7632), __byte_perm(v[2][e], v[3][e], 0x7632));
        }
      }
      if constexpr (TAIL > 0) {
        uint32_t v[4][2];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint2 x = *reinterpret_cast<const uint2*>(vr + (r ^ fx) * HD + FULL_I * 64 + g * 4);
          if (!FULL && !ok[r]) x = make_uint2(0u, 0u);
          v[r][0] = x.x;
          v[r][1] = x.y;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          pv(acc[8 * FULL_I + 2 * e], __byte_perm(v[0][e], v[1][e], 0x5410),
             __byte_perm(v[2][e], v[3][e], 0x5410));
          pv(acc[8 * FULL_I + 2 * e + 1], __byte_perm(v[0][e], v[1][e], 0x7632),
             __byte_perm(v[2][e], v[3][e], 0x7632));
        }
      }
    }
  }

  // The piece is complete: O of head g % G in acc[.][0..1] of lanes g < G.
  __device__ __forceinline__ void finish() {
    l += __shfl_xor_sync(0xFFFFFFFFu, l, 1);
    l += __shfl_xor_sync(0xFFFFFFFFu, l, 2);
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float hi = acc[n][i];
        float rest = acc[n][i + 2];
        if (G == 4) rest += __shfl_xor_sync(0xFFFFFFFFu, hi, 16);
        if (G == 2) rest = __shfl_xor_sync(0xFFFFFFFFu, hi, 8) + __shfl_xor_sync(0xFFFFFFFFu, hi, 16);
        acc[n][i] = fabsf(hi) < INFINITY ? hi + rest : hi;
      }
  }

  // f(offset in a row of HD, 8 consecutive outputs) for this lane's outputs
  template <typename F>
  __device__ __forceinline__ void each_vec(int t, F f) const {
    float v[8];
#pragma unroll
    for (int i = 0; i < FULL_I; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = acc[8 * i + e][h];
        f(64 * i + 16 * t + 8 * h, v);
      }
    if constexpr (TAIL > 0) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = acc[8 * FULL_I + (e & 3)][e >> 2];
      f(64 * FULL_I + 8 * t, v);
    }
  }
  // The G output rows, normalised.
  __device__ __forceinline__ void write_rows(T* rows, int lane) const {
    const int g = g_of(lane);
    if (g >= G) return;
    const float inv = l > 0.f ? 1.f / l : 0.f;
    each_vec(lane & 3, [&](int off, const float (&v)[8]) {
      *reinterpret_cast<uint4*>(rows + g * HD + off) =
          make_uint4(pack_bf16(v[0] * inv, v[1] * inv), pack_bf16(v[2] * inv, v[3] * inv),
                     pack_bf16(v[4] * inv, v[5] * inv), pack_bf16(v[6] * inv, v[7] * inv));
    });
  }
  // A partial state: G x HD unnormalised outputs, then (max, sum) per head.
  __device__ __forceinline__ void store_state(float* rec, int lane) const {
    const int g = g_of(lane);
    if (g >= G) return;
    each_vec(lane & 3, [&](int off, const float (&v)[8]) {
      float4* d = reinterpret_cast<float4*>(rec + g * HD + off);
      d[0] = make_float4(v[0], v[1], v[2], v[3]);
      d[1] = make_float4(v[4], v[5], v[6], v[7]);
    });
    if ((lane & 3) == 0) *reinterpret_cast<float2*>(rec + G * HD + 2 * g) = make_float2(m, l);
  }
};

}  // namespace attn_detail
}  // namespace wm
