// The cross-layer KV pool for a decode batch (Sec. 3.1 Steps 1-2), appended
// to the paged cache (Sec. 3.2).
//
// Kernels, in launch order:
//   1. prenorm   : per (token, layer) inverse RMS of h_l; writes the router
//                  input xi = [hhat_{L-1}, hhat_{L-1-p}, ...] for both branches;
//                  per token the RoPE cos/sin at pos = slot - 1.
//   2. router    : z = Wr[X] xi (split over the L'D reduction), fp32 partials;
//                  tcgen05 for bf16 (proj_tc.cu, proj_rows.cu), FMA for fp32.
//   3. mix       : alpha = reshape(z + br), htilde_j = sum_l alpha[j][l] hhat_l;
//                  bf16: on the tensor cores, the operand is htilde_j times the
//                  RMSNorm_j gain and the sum of squares goes to the projection's
//                  epilogue, which scales by 1/RMS; fp32: RMSNorm_j here.
//   4. projection: W^X_j x^X_j for every branch and channel; for bf16 on
//                  tcgen05 with the epilogue fused (proj_tc.cu, proj_rows.cu).
//   5. epilogue  : (fp32) keys: per-head QK-norm then RoPE; keys and values
//                  are written to the token's cache slot.
// The kernels are launched with programmatic dependent launch (but gemm_wxT_simt, see
// launch_gemm_f32) and wait for their predecessor with griddepcontrol.wait before they
// read anything but weights.
#include <math.h>

#include <utility>

#include "common.cuh"
#include "internal.h"

namespace wm {

namespace {

constexpr int kMixThreads = 256;
constexpr int kChanGroup = 4; // channels mixed per CTA
constexpr int kVecPerThread = 2;  // 8-element vectors per thread: D <= 256*8*2
// Token counts from which the fp32 pool runs its batched form of the mix (prefill
// groups): several tokens per CTA.  Below it (decode steps) one token per CTA
// spreads the few tokens over more SMs.
constexpr int kBatchedTokens = 64;
constexpr int kMixCG = 8;     // channels per CTA in the batched mix
constexpr int kMixLC = 8;     // most layers per staged chunk of h in the batched mix
constexpr size_t kMixStageBudget = 160 * 1024;  // shared memory for the staged chunks

// 16-byte asynchronous global -> shared copies (no registers held while in flight)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// PDL: may start before its predecessor has ended.
template <bool PDL = true, typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = PDL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// 8 consecutive elements as fp32 (one 16-byte load for bf16, two for fp32)
template <typename T>
__device__ __forceinline__ void load8f(const T* src, float* f);
template <>
__device__ __forceinline__ void load8f<float>(const float* src, float* f) {
  const float4 a = *reinterpret_cast<const float4*>(src);
  const float4 c = *reinterpret_cast<const float4*>(src + 4);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
  f[4] = c.x; f[5] = c.y; f[6] = c.z; f[7] = c.w;
}
template <>
__device__ __forceinline__ void load8f<__nv_bfloat16>(const __nv_bfloat16* src, float* f) {
  Elem<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4*>(src), f);
}
template <typename T>
__device__ __forceinline__ void store8f(T* dst, const float* f);
template <>
__device__ __forceinline__ void store8f<float>(float* dst, const float* f) {
  *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
  *reinterpret_cast<float4*>(dst + 4) = make_float4(f[4], f[5], f[6], f[7]);
}
template <>
__device__ __forceinline__ void store8f<__nv_bfloat16>(__nv_bfloat16* dst, const float* f) {
  uint4 u;
  __nv_bfloat162 t;
  t = __floats2bfloat162_rn(f[0], f[1]); u.x = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[2], f[3]); u.y = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[4], f[5]); u.z = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[6], f[7]); u.w = *reinterpret_cast<uint32_t*>(&t);
  *reinterpret_cast<uint4*>(dst) = u;
}

// ---------------------------------------------------------------- prenorm
// WPR warps per (token, layer) row; a lane keeps its part of the row (at most four
// 8-element vectors) in registers between the sum of squares and the two router
// inputs, so the row is read once, 16 bytes at a time.  Bound by memory and, in a
// decode step, by the latency of that one read (the kernel it replaces read 2
// bytes per load, twice: 17 us at 32 tokens, L = 32, D = 4096; this one: 7 us).
constexpr int kPrenormWarps = 4;

template <typename T, int WPR>
__global__ void __launch_bounds__(kPrenormWarps * 32) prenorm_kernel(const MixParams p) {
  constexpr int MAXV = 4;
  __shared__ float red[kPrenormWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * (kPrenormWarps / WPR) + warp / WPR;  // b * L + l
  const int u = (warp % WPR) * 32 + lane, nu = WPR * 32;            // thread of the row
  pdl_wait();
  const bool there = row < p.B * p.L;
  if (WPR == 1 && !there) return;
  const int b = row / p.L, l = row % p.L;
  const int nvec = there ? p.D / 8 : 0;
  const T* hp = reinterpret_cast<const T*>(p.h) + (int64_t)row * p.D;
  float f[MAXV][8], ss = 0.f;
#pragma unroll
  for (int v = 0; v < MAXV; ++v) {
    const int vi = u + v * nu;
    if (vi < nvec) load8f<T>(hp + vi * 8, f[v]);
    else
#pragma unroll
      for (int i = 0; i < 8; ++i) f[v][i] = 0.f;
  }
#pragma unroll
  for (int v = 0; v < MAXV; ++v)
#pragma unroll
    for (int i = 0; i < 8; ++i) ss = fmaf(f[v][i], f[v][i], ss);
  ss = warp_sum(ss);
  if (WPR > 1) {
    if (lane == 0) red[warp] = ss;
    __syncthreads();
    ss = 0.f;
#pragma unroll
    for (int w = 0; w < WPR; ++w) ss += red[warp / WPR * WPR + w];
    if (!there) return;
  }
  const float r = rsqrtf(ss / (float)p.D + p.eps_rms);
  if (u == 0) p.inv_rms[row] = r;
  const int from_top = p.L - 1 - l;
  if (from_top % p.p == 0) {  // router input block m holds layer L-1-m*p
    const int m = from_top / p.p;
#pragma unroll
    for (int X = 0; X < 2; ++X) {
      const T* g = reinterpret_cast<const T*>(p.pre_g[X]);
      T* xo = reinterpret_cast<T*>(p.xi) + ((int64_t)X * p.B + b) * ((int64_t)p.Lp * p.D) +
              (int64_t)m * p.D;
#pragma unroll
      for (int v = 0; v < MAXV; ++v) {
        const int vi = u + v * nu;
        if (vi >= nvec) break;
        float gv[8], o[8];
        load8f<T>(g + vi * 8, gv);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = f[v][i] * r * gv[i];
        store8f<T>(xo + vi * 8, o);
      }
    }
  }
  if (l == 0) {
    // RoPE angle pos * theta^(-2i/d) in fp64, reduced to [-pi, pi] before sincosf
    // (fp64 is slow here: a product with 1/2pi, not a division)
    const double pos = (double)(p.slot[b] - 1);
    for (int i = u; i < p.d / 2; i += nu) {
      const double a = pos * p.inv_freq[i];
      const double two_pi = 6.283185307179586476925286766559;
      const double inv_two_pi = 0.15915494309189533576888376337251;
      const float ar = (float)(a - two_pi * rint(a * inv_two_pi));
      float sn, cs;
      sincosf(ar, &sn, &cs);
      p.rope_cs[((int64_t)b * (p.d / 2) + i) * 2] = cs;
      p.rope_cs[((int64_t)b * (p.d / 2) + i) * 2 + 1] = sn;
    }
  }
}

// ---------------------------------------------------------------- W x^T (SIMT)
// out[z][n][m] = sum_{k in split} W[m][k] * X[n][k], z = batch * nsplit + split.
// Weights of batch item `bi` start at W[bi / per_branch] + (bi % per_branch) * w_stride.
constexpr int BM = 64, BN = 32, BK = 32;

struct GemmArgs {
  const void* W[2];
  int64_t w_stride;      // elements between consecutive items of one branch
  int per_branch;        // batch items per branch
  const void* X;         // [batch][N][K]
  int64_t x_stride;      // elements between batch items of X
  float* out;            // [batch][nsplit][N][M]
  int M, N, K, nsplit, k_per_split;
};

__global__ void __launch_bounds__(256) gemm_wxT_simt(const GemmArgs a) {
  __shared__ float Ws[BK][BM + 4];
  __shared__ float Xs[BK][BN + 4];
  const int split = blockIdx.z % a.nsplit, bi = blockIdx.z / a.nsplit;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int kbeg = split * a.k_per_split;
  const int kend = min(a.K, kbeg + a.k_per_split);
  const float* W = reinterpret_cast<const float*>(a.W[bi / a.per_branch]) +
                (int64_t)(bi % a.per_branch) * a.w_stride;
  const float* X = reinterpret_cast<const float*>(a.X) + (int64_t)bi * a.x_stride;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  pdl_wait();
  float acc[4][2] = {};
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
    {  // W tile: row tid/4, 8 consecutive k
      const int r = tid >> 2, kk = (tid & 3) * 8;
      const int m = m0 + r, k = k0 + kk;
      float f[8];
      if (m < a.M && k + 8 <= kend) {
        load8f<float>(W + (int64_t)m * a.K + k, f);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          f[i] = (m < a.M && k + i < kend) ? ldf(W + (int64_t)m * a.K + k + i) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) Ws[kk + i][r] = f[i];
    }
    {  // X tile: token tid/8, 4 consecutive k
      const int n = tid >> 3, kk = (tid & 7) * 4;
      const int nn = n0 + n, k = k0 + kk;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        Xs[kk + i][n] = (nn < a.N && k + i < kend) ? ldf(X + (int64_t)nn * a.K + k + i) : 0.f;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      const float4 w = *reinterpret_cast<const float4*>(&Ws[kk][tx * 4]);
      const float2 x = *reinterpret_cast<const float2*>(&Xs[kk][ty * 2]);
      acc[0][0] = fmaf(w.x, x.x, acc[0][0]);
      acc[1][0] = fmaf(w.y, x.x, acc[1][0]);
      acc[2][0] = fmaf(w.z, x.x, acc[2][0]);
      acc[3][0] = fmaf(w.w, x.x, acc[3][0]);
      acc[0][1] = fmaf(w.x, x.y, acc[0][1]);
      acc[1][1] = fmaf(w.y, x.y, acc[1][1]);
      acc[2][1] = fmaf(w.z, x.y, acc[2][1]);
      acc[3][1] = fmaf(w.w, x.y, acc[3][1]);
    }
    __syncthreads();
  }
  float* out = a.out + (int64_t)blockIdx.z * a.N * a.M;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int n = n0 + ty * 2 + j;
    if (n >= a.N) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + tx * 4 + i;
      if (m < a.M) out[(int64_t)n * a.M + m] = acc[i][j];
    }
  }
}

// The same product for few tokens of fp32: a decode step of a small batch reads
// every weight once for a handful of multiply-adds, so it is a stream of W (and,
// at small sizes, one chain of load latencies).  A warp takes R weight rows at a
// time against NT tokens, a lane every 32nd 16-byte vector of them, U of each row
// in flight and the next U requested before these are used; the first ones before
// the dependency wait (no kernel of the step writes weights), and past L1.  The
// tokens' vectors come through L1, which the CTA's warps share; with more tokens
// than NT the CTAs of all token groups of a row block are neighbours, so W comes
// from HBM once.  Four rows where a token group is wide: that halves the loads of
// tokens, which bind there.  The tiled kernel above, two barriers per 32 elements
// of K and ceil(M / 64) CTAs per split, has 32 tokens in a tile whatever their
// number: the line lies where it is as fast.  Pools (us, tiled / streamed; L = k = 16,
// D = 512, 3 heads of 96, then L = 32, k = 16, D = 4096, 32 heads of 128): one token
// 70 / 21 and 2061 / 394; 8 tokens 145 / 29 and 2076 / 709; 16 tokens 134 / 39 and
// 2096 / 1199.
constexpr int kGemvTokens = 16;
constexpr int kGemvWarps = 4;

template <int NT, int R, int U>
__global__ void __launch_bounds__(kGemvWarps * 32) gemv_wxT_f32(const GemmArgs a) {
  constexpr int STEP = 32 * 4;
  const int split = blockIdx.z % a.nsplit, bi = blockIdx.z / a.nsplit;
  const int lane = threadIdx.x & 31;
  const int groups = (a.N + NT - 1) / NT, n0 = (int)blockIdx.x % groups * NT;  // this CTA's tokens
  const int m0 = ((int)blockIdx.x / groups * kGemvWarps + (threadIdx.x >> 5)) * R;
  const int kend = min(a.K, (split + 1) * a.k_per_split);
  int k = split * a.k_per_split + lane * 4;
  const float* W = reinterpret_cast<const float*>(bi < a.per_branch ? a.W[0] : a.W[1]) +
                   (int64_t)(bi % a.per_branch) * a.w_stride;
  const float* X = reinterpret_cast<const float*>(a.X) + (int64_t)bi * a.x_stride + (int64_t)n0 * a.K;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool live = m0 < a.M;
  auto load_w = [&](float4 (&w)[U][R], int k0) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int kk = k0 + u * STEP;
        w[u][r] = live && m0 + r < a.M && kk < kend
                      ? __ldcg(reinterpret_cast<const float4*>(W + (int64_t)(m0 + r) * a.K + kk))
                      : zero;
      }
  };
  float4 w[U][R], wn[U][R];
  load_w(w, k);
  pdl_wait();
  if (!live) return;
  float acc[R][NT];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int t = 0; t < NT; ++t) acc[r][t] = 0.f;
  // (the bound is the warp's, so that lanes past the split's end stay with it: their weights are 0)
  for (; k - lane * 4 < kend; k += U * STEP) {
    load_w(wn, k + U * STEP);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int kk = k + u * STEP;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const float4 x = kk < kend && n0 + t < a.N
                             ? *reinterpret_cast<const float4*>(X + (int64_t)t * a.K + kk)
                             : zero;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          acc[r][t] = fmaf(w[u][r].x, x.x, acc[r][t]);
          acc[r][t] = fmaf(w[u][r].y, x.y, acc[r][t]);
          acc[r][t] = fmaf(w[u][r].z, x.z, acc[r][t]);
          acc[r][t] = fmaf(w[u][r].w, x.w, acc[r][t]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) w[u][r] = wn[u][r];
  }
  float* out = a.out + (int64_t)blockIdx.z * a.N * a.M;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const float v = warp_sum(acc[r][t]);
      if (lane == 0 && n0 + t < a.N && m0 + r < a.M) out[(int64_t)(n0 + t) * a.M + m0 + r] = v;
    }
}

// out[batch][split][n][m] = sum over the split's k of W[m][k] X[n][k]
cudaError_t launch_gemm_f32(const GemmArgs& a, int batch, cudaStream_t s) {
  const unsigned z = (unsigned)(batch * a.nsplit);
  if (a.N <= kGemvTokens) {
    auto go = [&](auto kern, int nt, int r) {
      const int rows = kGemvWarps * r, groups = (a.N + nt - 1) / nt;
      return launch_pdl(kern, dim3((unsigned)((a.M + rows - 1) / rows * groups), 1, z), dim3(kGemvWarps * 32),
                        0, s, a);
    };
    if (a.N == 1) return go(gemv_wxT_f32<1, 2, 4>, 1, 2);
    if (a.N == 2) return go(gemv_wxT_f32<2, 2, 4>, 2, 2);
    if (a.N <= 4) return go(gemv_wxT_f32<4, 4, 2>, 4, 4);
    return go(gemv_wxT_f32<8, 4, 2>, 8, 4);
  }
  // Without programmatic launch: placed while the predecessor runs, the few tiles land
  // side by side on the SMs that have room, and the product takes two or three times as
  // long (pool of L = 16, k = 8, D = 1024, 8 heads of 64: 227-302 us at 32 tokens, by what
  // the kernels before it look like; 105 so; 257 and 137 at 64, 394 and 199 at 128).
  return launch_pdl<false>(gemm_wxT_simt, dim3((a.M + BM - 1) / BM, (a.N + BN - 1) / BN, z), dim3(256),
                           0, s, a);
}

// ---------------------------------------------------------------- mix (bf16)
// Per token and branch, htilde = (alpha r) H with alpha [k][L] (r_l = 1/RMS of
// layer l folded in) and H [L][D] the token's states: a contraction, so it runs
// on the tensor cores, m16n8k16 with channels as M, layers as K and 8 elements
// of D as N (the matrices are per token and 16 wide: too small for tcgen05's
// 128-row tiles).  The states are bf16 as they are; alpha stays fp32 by being
// three bf16 terms of 8 bits each, three MMAs into one fp32 accumulator, so
// products and sums are those of fp32 arithmetic.  The pre-mix gain g, a factor
// per element, multiplies the sum.
//
// A unit is one token and one part of D; a warp takes 64 elements at a time for
// both branches, so h is read once per 16 channels.  Lane (t = lane % 4, g =
// lane / 4) loads 16 bytes of layers 2t, 2t+1, 2t+8, 2t+9 at vector v(g); element
// i of the vectors is column g of MMA i, so the eight MMAs' results of one column
// are 8 consecutive elements, one 16-byte store, and the four t of a store cover
// 64 bytes.  RMSNorm_j's 1/RMS is left to the projection's epilogue (it is one
// factor per token and channel), so parts of D need not meet.  Decode steps and
// small groups (COOP): a CTA per unit, its warps share the sum of the router's many
// split partials and a warp has one or a few 64-element steps.  Large groups of
// tokens (mix_token_warps): a warp per unit, nothing shared, the next step's states
// in flight while this step's are used (as CTAs, which wait for them, 75 us at the
// 4096 tokens below).
//
// Bound by memory: h in, the operand out (201 MB at 4096 tokens, L = k = 16, D =
// 512).  There the scalar kernel before took 194 us, this one 59; at 32
// tokens, L = 32, k = 16, D = 4096: 40 and 18 (cold caches).
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_16816_first(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// alpha[j][l] r_l of one token, branch X, for N (j, l) pairs: (bias + the router's
// split partials) r_l, 0 outside.  The N loads of a split are in flight together.
template <int N>
__device__ __forceinline__ void mix_alpha(const MixParams& p, int b, int X, const int (&j)[N],
                                          const int (&l)[N], float (&a)[N]) {
  const int kL = p.k * p.L;
  const float* zp = p.zpart + ((int64_t)X * p.nsplit_r * p.B + b) * kL;
  const __nv_bfloat16* br = reinterpret_cast<const __nv_bfloat16*>(p.br[X]);
  int o[N];
  float r[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const bool in = j[i] < p.k && l[i] < p.L;
    o[i] = in ? j[i] * p.L + l[i] : 0;
    r[i] = in ? p.inv_rms[b * p.L + l[i]] : 0.f;
    a[i] = in ? __bfloat162float(br[o[i]]) : 0.f;
  }
#pragma unroll(N > 2 ? 2 : 8)
  for (int s = 0; s < p.nsplit_r; ++s, zp += (int64_t)p.B * kL)
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] += zp[o[i]];
#pragma unroll
  for (int i = 0; i < N; ++i) a[i] = j[i] < p.k && l[i] < p.L ? a[i] * r[i] : 0.f;
}

constexpr int kCoopWarps = 8, kTokenWarps = 4;  // warps per CTA

// KSR: blocks of 16 layers whose states a warp keeps in registers (L <= 16 KSR);
// 0: any L, the states read again for the second branch.
template <bool COOP, int KSR>
__global__ void __launch_bounds__((COOP ? kCoopWarps : kTokenWarps) * 32, COOP ? 2 : KSR == 2 ? 3 : 4)
    mix_mma_kernel(const MixParams p, int ks_count, int csteps) {
  const int KS = KSR > 0 ? KSR : ks_count;
  constexpr int KB = KSR > 0 ? KSR : 1;
  constexpr int NW = COOP ? kCoopWarps : kTokenWarps;
  // alpha of 16 channels in the MMA's operand layout, [X][KS][3 terms][32 lanes]
  // (one for the CTA, or one per warp), then (COOP) sums of squares [warps][X][16]
  extern __shared__ uint4 frag_s[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4* frag = frag_s + (COOP ? 0 : warp * 2 * KS * 3 * 32);
  float* wss = reinterpret_cast<float*>(frag_s + 2 * KS * 3 * 32);
  const int nparts = p.mix_parts;
  const int unit = COOP ? (int)blockIdx.x : (int)blockIdx.x * NW + warp;
  const int b = unit / nparts, part = unit - b * nparts;
  const int t = lane & 3, g = lane >> 2;
  const int L = p.L, nvec = p.D / 8;
  const int vg = (g >> 1) + 4 * (g & 1);  // the vector lane column g stands for
  const int c0 = part * csteps + (COOP ? warp : 0), cstep = COOP ? NW : 1;
  const int c_end = min((nvec + 7) / 8, (part + 1) * csteps);
  if (COOP) {  // gains and (a hint: the data may still be on its way) states towards L2
    for (int i = tid; i < (p.k + 1) * 2 * (c_end - part * csteps); i += NW * 32) {
      const int c = part * csteps + i / ((p.k + 1) * 2), r = i % ((p.k + 1) * 2);
      const __nv_bfloat16* q = reinterpret_cast<const __nv_bfloat16*>(r < 2 ? p.pre_g[r] : p.ch_g[r & 1]);
      if (c * 64 < p.D) prefetch_l2(q + (r < 2 ? 0 : (int64_t)((r - 2) >> 1) * p.D) + c * 64);
    }
  }
  pdl_wait();
  if (!COOP && b >= p.B) return;  // (no block barrier below)
  const __nv_bfloat16* hp = reinterpret_cast<const __nv_bfloat16*>(p.h) + (int64_t)b * L * p.D;
  // 16 bytes of the lane's four layers of block ks, step c
  auto load_h = [&](int c, int ks, uint4 (&hv)[4]) {
    const int vi = c * 8 + vg;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int l = ks * 16 + 2 * t + (q & 1) + 8 * (q >> 1);
      hv[q] = c < c_end && l < L && vi < nvec
                  ? __ldcg(reinterpret_cast<const uint4*>(hp + (int64_t)l * p.D + vi * 8))
                  : make_uint4(0, 0, 0, 0);
    }
  };

  for (int mt = blockIdx.y; mt * 16 < p.k; mt += gridDim.y) {
    uint4 hn[KB][4];
    if (KSR > 0)
#pragma unroll
      for (int ks = 0; ks < KB; ++ks) load_h(c0, ks, hn[ks]);
    if (COOP) {
      if (mt > (int)blockIdx.y) __syncthreads();
      // the layer pairs and channels there are; the rest of the operand is 0
      const int npair = (L + 1) / 2, nch = min(16, p.k - mt * 16);
      if (npair < KS * 8 || nch < 16) {
        for (int i = tid; i < 2 * KS * 3 * 32; i += NW * 32) frag[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
      }
      for (int i = tid; i < 2 * nch * npair; i += NW * 32) {  // two layers at a time
        const int lp = i % npair, rem = i / npair, jj = rem % nch, X = rem / nch;
        float a[2];
        mix_alpha<2>(p, b, X, {mt * 16 + jj, mt * 16 + jj}, {2 * lp, 2 * lp + 1}, a);
        // operand register and lane of row jj, columns l % 16 and l % 16 + 1
        const int reg = (jj >> 3) + 2 * ((lp >> 2) & 1), ln = (jj & 7) * 4 + (lp & 3);
        uint32_t* f = reinterpret_cast<uint32_t*>(frag + (X * KS + (lp >> 3)) * 3 * 32);
#pragma unroll
        for (int s = 0; s < 3; ++s) {  // the next 8 bits of each
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(a[0], a[1]);
          a[0] -= __bfloat162float(h2.x);
          a[1] -= __bfloat162float(h2.y);
          f[(s * 32 + ln) * 4 + reg] = *reinterpret_cast<const uint32_t*>(&h2);
        }
      }
      __syncthreads();
    } else {
      __syncwarp();
      for (int i = 0; i < 2 * KS; ++i) {  // X = i / KS, layer block i % KS
        const int X = i / KS, ks = i - X * KS;
        float a[8];  // operand registers r: rows g, g + 8; columns 2t, 2t+1 and + 8
        int jj[8], ll[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          jj[r] = mt * 16 + g + 8 * ((r >> 1) & 1);
          ll[r] = ks * 16 + 2 * t + (r & 1) + 8 * (r >> 2);
        }
        mix_alpha<8>(p, b, X, jj, ll, a);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          uint32_t w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(a[2 * r], a[2 * r + 1]);
            a[2 * r] -= __bfloat162float(h2.x);
            a[2 * r + 1] -= __bfloat162float(h2.y);
            w[r] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          frag[(i * 3 + s) * 32 + lane] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      __syncwarp();
    }

    float ss[2][2] = {};  // [X][channel g, g + 8]
    for (int c = c0; c < c_end; c += cstep) {
      uint32_t bf[KB][8][2];  // element i of layers (2t, 2t+1) and (2t+8, 2t+9)
      auto pack = [&](const uint4 (&hv)[4], uint32_t (&f)[8][2]) {
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const uint32_t lo[4] = {hv[2 * h2].x, hv[2 * h2].y, hv[2 * h2].z, hv[2 * h2].w};
          const uint32_t hi[4] = {hv[2 * h2 + 1].x, hv[2 * h2 + 1].y, hv[2 * h2 + 1].z, hv[2 * h2 + 1].w};
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            f[2 * w][h2] = __byte_perm(lo[w], hi[w], 0x5410);
            f[2 * w + 1][h2] = __byte_perm(lo[w], hi[w], 0x7632);
          }
        }
      };
      if (KSR > 0) {
#pragma unroll
        for (int ks = 0; ks < KB; ++ks) {
          pack(hn[ks], bf[ks]);
          if (!COOP) load_h(c + cstep, ks, hn[ks]);  // in flight behind this step's work
        }
      }
#pragma unroll
      for (int X = 0; X < 2; ++X) {
        const __nv_bfloat16* pg = reinterpret_cast<const __nv_bfloat16*>(p.pre_g[X]);
        const __nv_bfloat16* cg = reinterpret_cast<const __nv_bfloat16*>(p.ch_g[X]);
        __nv_bfloat16* xop = reinterpret_cast<__nv_bfloat16*>(p.xop);
        // gains of this lane's outputs (column 2t + q: vector t + 4q; channels g, g
        // + 8), through the read-only path: not held up by the stores
        uint4 gr[2], cr[2][2];
        const int v0 = c * 8 + t;
        const int jr[2] = {mt * 16 + g, mt * 16 + g + 8};
        const bool in[2] = {v0 < nvec, v0 + 4 < nvec}, ch[2] = {jr[0] < p.k, jr[1] < p.k};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          gr[q] = in[q] ? __ldg(reinterpret_cast<const uint4*>(pg) + v0 + 4 * q) : make_uint4(0, 0, 0, 0);
#pragma unroll
          for (int r = 0; r < 2; ++r)
            cr[q][r] = in[q] && ch[r] ? __ldg(reinterpret_cast<const uint4*>(cg + (int64_t)jr[r] * p.D) + v0 + 4 * q)
                                      : make_uint4(0, 0, 0, 0);
        }
        float acc[8][4];
        for (int ks = 0; ks < KS; ++ks) {
          if (KSR == 0) {
            uint4 hv[4];
            load_h(c, ks, hv);
            pack(hv, bf[0]);
          }
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            const uint4 a = frag[((X * KS + ks) * 3 + s) * 32 + lane];
            const uint32_t(&f)[8][2] = bf[KSR > 0 ? ks : 0];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if (ks == 0 && s == 0) mma_16816_first(acc[i], a, f[i][0], f[i][1]);
              else mma_16816(acc[i], a, f[i][0], f[i][1]);
            }
          }
        }
        float2 gv[8];  // of both columns, as pairs like the accumulators
        {
          float x0[8], x1[8];
          Elem<__nv_bfloat16>::unpack(gr[0], x0);
          Elem<__nv_bfloat16>::unpack(gr[1], x1);
#pragma unroll
          for (int i = 0; i < 8; ++i) gv[i] = make_float2(x0[i], x1[i]);
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float x0[8], x1[8];
          Elem<__nv_bfloat16>::unpack(cr[0][r], x0);
          Elem<__nv_bfloat16>::unpack(cr[1][r], x1);
          float2 s2 = make_float2(0.f, 0.f);
          float o0[8], o1[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 y = __fmul2_rn(make_float2(acc[i][2 * r], acc[i][2 * r + 1]), gv[i]);
            s2 = __ffma2_rn(y, y, s2);
            const float2 o = __fmul2_rn(y, make_float2(x0[i], x1[i]));
            o0[i] = o.x;
            o1[i] = o.y;
          }
          if (in[0]) ss[X][r] += s2.x;  // (a column past D holds zero times whatever: skipped)
          if (in[1]) ss[X][r] += s2.y;
          if (ch[r]) {
            __nv_bfloat16* dst = xop + (((int64_t)X * p.k + jr[r]) * p.B + b) * p.D + v0 * 8;
            if (in[0]) store8f<__nv_bfloat16>(dst, o0);
            if (in[1]) store8f<__nv_bfloat16>(dst + 32, o1);
          }
        }
      }
      if (COOP && KSR > 0 && c + cstep < c_end) {  // (few steps a warp: no second set of registers)
#pragma unroll
        for (int ks = 0; ks < KB; ++ks) load_h(c + cstep, ks, hn[ks]);
      }
    }
    // sums of squares: over the four t of a channel, and the CTA's warps
#pragma unroll
    for (int X = 0; X < 2; ++X)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float v = ss[X][r];
        v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
        v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
        if (t != 0) continue;
        const int j = mt * 16 + g + 8 * r;
        if (COOP)
          wss[(warp * 2 + X) * 16 + g + 8 * r] = v;
        else if (j < p.k)
          p.ssq[(((int64_t)X * p.k + j) * nparts + part) * p.B + b] = v;
      }
    if (COOP) {
      __syncthreads();
      if (tid < 32) {
        const int X = tid >> 4, j = mt * 16 + (tid & 15);
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) v += wss[(w * 2 + X) * 16 + (tid & 15)];
        if (j < p.k) p.ssq[(((int64_t)X * p.k + j) * nparts + part) * p.B + b] = v;
      }
    }
  }
}

// ---------------------------------------------------------------- mix (fp32)
// One CTA per (token, branch, group of kChanGroup channels).  Thread t owns
// the 8-element vectors t, t + 256 of D, so h, gains and the output move as
// 16-byte vectors.
__global__ void __launch_bounds__(kMixThreads) mix_kernel(const MixParams p) {
  extern __shared__ float sm[];  // alpha[kChanGroup][L], r[L]
  __shared__ float red[kMixThreads / 32][kChanGroup];
  float* alpha = sm;
  float* rl = sm + kChanGroup * p.L;
  const int b = blockIdx.x, X = blockIdx.y, j0 = blockIdx.z * kChanGroup;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nj = min(kChanGroup, p.k - j0);
  const int kL = p.k * p.L;
  const int nvec = p.D / 8;
  const float* hp = reinterpret_cast<const float*>(p.h) + (int64_t)b * p.L * p.D;
  const float* g = reinterpret_cast<const float*>(p.pre_g[X]);
  pdl_wait();
  const float* br = reinterpret_cast<const float*>(p.br[X]);
  // alpha[j][l] = z[j*L + l] = bias + sum of the router's split partials
  for (int i = tid; i < nj * p.L; i += kMixThreads) {
    const int o = j0 * p.L + i;
    const float* zp = p.zpart + ((int64_t)X * p.nsplit_r * p.B + b) * kL + o;
    float z = ldf(br + o);
#pragma unroll 8
    for (int s2 = 0; s2 < p.nsplit_r; ++s2) z += zp[(int64_t)s2 * p.B * kL];
    alpha[i] = z;
  }
  for (int i = tid; i < p.L; i += kMixThreads) rl[i] = p.inv_rms[b * p.L + i];
  __syncthreads();

  float gv[kVecPerThread][8];
  float acc[kChanGroup][kVecPerThread][8];
#pragma unroll
  for (int v = 0; v < kVecPerThread; ++v) {
    const int vi = tid + v * kMixThreads;
    if (vi < nvec) load8f<float>(g + vi * 8, gv[v]);
#pragma unroll
    for (int jj = 0; jj < kChanGroup; ++jj)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[jj][v][i] = 0.f;
  }
#pragma unroll 4
  for (int l = 0; l < p.L; ++l) {
    const float r = rl[l];
    float a[kChanGroup];
#pragma unroll
    for (int jj = 0; jj < kChanGroup; ++jj) a[jj] = jj < nj ? alpha[jj * p.L + l] : 0.f;
#pragma unroll
    for (int v = 0; v < kVecPerThread; ++v) {
      const int vi = tid + v * kMixThreads;
      if (vi < nvec) {
        float hv[8];
        load8f<float>(hp + (int64_t)l * p.D + vi * 8, hv);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float hh = hv[i] * r * gv[v][i];  // pre-mix RMSNorm with gain
#pragma unroll
          for (int jj = 0; jj < kChanGroup; ++jj) acc[jj][v][i] = fmaf(a[jj], hh, acc[jj][v][i]);
        }
      }
    }
  }
  // per-channel sums of squares, reduced over the block for all channels at once
  float ss[kChanGroup];
#pragma unroll
  for (int jj = 0; jj < kChanGroup; ++jj) {
    float t = 0.f;
#pragma unroll
    for (int v = 0; v < kVecPerThread; ++v)
#pragma unroll
      for (int i = 0; i < 8; ++i) t = fmaf(acc[jj][v][i], acc[jj][v][i], t);
    t = warp_sum(t);
    if (lane == 0) red[warp][jj] = t;
  }
  __syncthreads();
#pragma unroll
  for (int jj = 0; jj < kChanGroup; ++jj) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kMixThreads / 32; ++w) t += red[w][jj];
    ss[jj] = rsqrtf(t / (float)p.D + p.eps_rms);
  }
  float* xop = reinterpret_cast<float*>(p.xop);
#pragma unroll
  for (int jj = 0; jj < kChanGroup; ++jj) {
    if (jj >= nj) break;
    const int j = j0 + jj;
    const float* cg = reinterpret_cast<const float*>(p.ch_g[X]) + (int64_t)j * p.D;
    float* xo = xop + (((int64_t)X * p.k + j) * p.B + b) * p.D;
#pragma unroll
    for (int v = 0; v < kVecPerThread; ++v) {
      const int vi = tid + v * kMixThreads;
      if (vi < nvec) {
        float cv[8], o[8];
        load8f<float>(cg + vi * 8, cv);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = acc[jj][v][i] * ss[jj] * cv[i];
        store8f<float>(xo + vi * 8, o);
      }
    }
  }
}

// Batched form: one CTA per (tb tokens, branch, kMixCG channels); tpt
// threads (whole warps) per token, thread u of a token owning the 8-element
// vectors u, u + tpt, ... of D.  alpha of the CTA's tokens is summed from the
// router's split partials once, into shared memory.  Each thread streams its
// own vectors of h through a private 2 x kMixLC-layer buffer in shared memory
// with asynchronous copies, so many loads are in flight without holding
// registers.
template <int VPT>
__global__ void __launch_bounds__(kMixThreads) mix_tokens_kernel(const MixParams p, int tpt, int tb,
                                                                  int lc) {
  // alpha[tb][kMixCG][L], rl[tb][L], red[warps][kMixCG], then (16-byte
  // aligned) the h staging buffers [2][lc][VPT][threads] of one vector
  // (8 elements: VB 16-byte units) each; lc <= kMixLC layers per chunk
  extern __shared__ float sm[];
  constexpr int VB = 8 * (int)sizeof(float) / 16;
  const int X = blockIdx.y, j0 = blockIdx.z * kMixCG;
  const int nj = min(kMixCG, p.k - j0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = tid / tpt, u = tid % tpt;
  const int b0 = blockIdx.x * tb, b = b0 + t;
  const bool live = t < tb && b < p.B;
  const int L = p.L, kL = p.k * p.L, nvec = p.D / 8;
  float* alpha = sm;
  float* rl = alpha + tb * kMixCG * L;
  float* red = rl + tb * L;
  uint4* hbuf = reinterpret_cast<uint4*>(
      (reinterpret_cast<uintptr_t>(red + (blockDim.x / 32) * kMixCG) + 15) & ~static_cast<uintptr_t>(15));
  const int nth = blockDim.x;
  auto hslot = [&](int stage, int l, int v) -> uint4* {
    return hbuf + (((stage * lc + l) * VPT + v) * nth + tid) * VB;
  };
  const float* hp = reinterpret_cast<const float*>(p.h) + (int64_t)b * L * p.D;
  // copies of layers [l0, l0 + lc) of this thread's vectors into `stage`
  auto stage_chunk = [&](int stage, int l0) {
    if (live)
      for (int l = l0; l < min(L, l0 + lc); ++l)
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
          const int vi = u + v * tpt;
          if (vi < nvec)
#pragma unroll
            for (int q = 0; q < VB; ++q)
              cp_async16(hslot(stage, l - l0, v) + q,
                         reinterpret_cast<const uint4*>(hp + (int64_t)l * p.D + vi * 8) + q);
        }
    cp_async_commit();
  };
  pdl_wait();
  stage_chunk(0, 0);
  stage_chunk(1, lc);
  const float* br = reinterpret_cast<const float*>(p.br[X]);
  for (int i = tid; i < tb * nj * L; i += blockDim.x) {
    const int tt = i / (nj * L), rem = i % (nj * L);
    const int bb = b0 + tt, o = j0 * L + rem;
    float z = 0.f;
    if (bb < p.B) {
      z = ldf(br + o);
      const float* zp = p.zpart + ((int64_t)X * p.nsplit_r * p.B + bb) * kL + o;
#pragma unroll 8
      for (int s2 = 0; s2 < p.nsplit_r; ++s2) z += zp[(int64_t)s2 * p.B * kL];
    }
    alpha[tt * kMixCG * L + rem] = z;  // [tt][jj][l] with jj = rem / L, l = rem % L
  }
  for (int i = tid; i < tb * L; i += blockDim.x) {
    const int bb = b0 + i / L;
    rl[i] = bb < p.B ? p.inv_rms[(int64_t)bb * L + i % L] : 0.f;
  }
  __syncthreads();

  const float* g = reinterpret_cast<const float*>(p.pre_g[X]);
  float gv[VPT][8];
  float acc[kMixCG][VPT][8];
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int vi = u + v * tpt;
    if (live && vi < nvec) load8f<float>(g + vi * 8, gv[v]);
#pragma unroll
    for (int jj = 0; jj < kMixCG; ++jj)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[jj][v][i] = 0.f;
  }
  {
    const float* al = alpha + t * kMixCG * L;
    for (int l0 = 0, c = 0; l0 < L; l0 += lc, ++c) {
      cp_async_wait<1>();  // this thread's copies of chunk c have landed
      for (int l = l0; l < min(L, l0 + lc); ++l) {
      if (!live) break;
      const float r = rl[t * L + l];
      float a[kMixCG];
#pragma unroll
      for (int jj = 0; jj < kMixCG; ++jj) a[jj] = jj < nj ? al[jj * L + l] : 0.f;
#pragma unroll
      for (int v = 0; v < VPT; ++v) {
        const int vi = u + v * tpt;
        if (vi < nvec) {
          float hv[8];
          load8f<float>(reinterpret_cast<const float*>(hslot(c & 1, l - l0, v)), hv);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float hh = hv[i] * r * gv[v][i];  // pre-mix RMSNorm with gain
#pragma unroll
            for (int jj = 0; jj < kMixCG; ++jj) acc[jj][v][i] = fmaf(a[jj], hh, acc[jj][v][i]);
          }
        }
      }
      }
      stage_chunk(c & 1, l0 + 2 * lc);  // refill the buffer just consumed
    }
    cp_async_wait<0>();
  }
  // per-channel sums of squares over the token's warps
#pragma unroll
  for (int jj = 0; jj < kMixCG; ++jj) {
    float q = 0.f;
#pragma unroll
    for (int v = 0; v < VPT; ++v)
#pragma unroll
      for (int i = 0; i < 8; ++i) q = fmaf(acc[jj][v][i], acc[jj][v][i], q);
    q = warp_sum(q);
    if (lane == 0) red[warp * kMixCG + jj] = q;
  }
  __syncthreads();
  if (!live) return;
  const int w0 = t * (tpt / 32), nw = tpt / 32;
  float* xop = reinterpret_cast<float*>(p.xop);
#pragma unroll
  for (int jj = 0; jj < kMixCG; ++jj) {
    if (jj >= nj) break;
    float q = 0.f;
    for (int w = 0; w < nw; ++w) q += red[(w0 + w) * kMixCG + jj];
    const float sc = rsqrtf(q / (float)p.D + p.eps_rms);
    const int j = j0 + jj;
    const float* cg = reinterpret_cast<const float*>(p.ch_g[X]) + (int64_t)j * p.D;
    float* xo = xop + (((int64_t)X * p.k + j) * p.B + b) * p.D;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
      const int vi = u + v * tpt;
      if (vi < nvec) {
        float cv[8], o[8];
        load8f<float>(cg + vi * 8, cv);
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = acc[jj][v][i] * sc * cv[i];
        store8f<float>(xo + vi * 8, o);
      }
    }
  }
}

// ---------------------------------------------------------------- epilogue
// fp32 path: one CTA per (token, channel, branch), a warp per kv head; lane t
// handles the RoPE pairs (i, i + HD/2) for i = t, t + 32, ...
template <int HD>
__global__ void __launch_bounds__(128) kv_epilogue_kernel(const MixParams p) {
  constexpr int HALF = HD / 2;
  constexpr int NP = (HALF + 31) / 32;
  const int b = blockIdx.x, j = blockIdx.y, X = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  const int s = p.slot[b];
  if (s < 1 || s >= p.max_pages * p.P) {
    if (threadIdx.x == 0 && j == 0 && X == 0) report(p.status, WM_ERR_BOUNDS);
    return;
  }
  const int pg = p.page_table[(int64_t)b * p.max_pages + (s >> p.log2P)];
  if (pg < 0 || pg >= p.num_pages) {
    if (threadIdx.x == 0 && j == 0 && X == 0) report(p.status, WM_ERR_BOUNDS);
    return;
  }
  const int nout = p.Hkv * HD;
  const float* src = p.proj + (((int64_t)X * p.k + j) * p.B + b) * nout;
  float* pool = reinterpret_cast<float*>(X == 0 ? p.k_pool : p.v_pool);
  const int64_t base = (((int64_t)j * p.num_pages + pg) * p.Hkv) * p.P + (s & (p.P - 1));
  const float* qg = reinterpret_cast<const float*>(p.qk_g) + (int64_t)j * HD;
  for (int hh = warp; hh < p.Hkv; hh += 4) {
    float y0[NP], y1[NP];
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      const int i = lane + 32 * t;
      y0[t] = i < HALF ? src[hh * HD + i] : 0.f;
      y1[t] = i < HALF ? src[hh * HD + i + HALF] : 0.f;
    }
    if (X == 0) {
      float ss = 0.f;
#pragma unroll
      for (int t = 0; t < NP; ++t) ss = fmaf(y0[t], y0[t], fmaf(y1[t], y1[t], ss));
      ss = warp_sum(ss);
      const float rr = rsqrtf(ss / (float)HD + p.eps_qk);
#pragma unroll
      for (int t = 0; t < NP; ++t) {
        const int i = lane + 32 * t;
        if (i < HALF) {
          const float x0 = y0[t] * rr * ldf(qg + i), x1 = y1[t] * rr * ldf(qg + i + HALF);
          const float cs = p.rope_cs[((int64_t)b * HALF + i) * 2];
          const float sn = p.rope_cs[((int64_t)b * HALF + i) * 2 + 1];
          y0[t] = x0 * cs - x1 * sn;  // rotate-half RoPE
          y1[t] = x1 * cs + x0 * sn;
        }
      }
    }
    float* dst = pool + (base + (int64_t)hh * p.P) * HD;
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      const int i = lane + 32 * t;
      if (i < HALF) {
        dst[i] = Elem<float>::from_f(y0[t]);
        dst[i + HALF] = Elem<float>::from_f(y1[t]);
      }
    }
  }
}

// Does the bf16 mix give every token to one warp (mix_mma_kernel without COOP)?  It pays
// once there are enough tokens to fill the SMs with warps and few router splits, which
// each warp sums by itself: below, a CTA per token or part of one.  Layers of two
// blocks, whose next states the warp form keeps in flight, sooner.  Whole pools (us, CTA
// form / warp form), L = 16, k = 16, D = 1024, 8 heads of 128: 49 / 60 at 128 tokens, 85
// / 97 at 512, 136 / 159 at 1024, 210 / 218 at 1536, 247 / 247 at 2048; L = 32, k = 4, D
// = 2048, 8 heads of 128: 67 / 110, 126 / 144, 223 / 204, 311 / 273, 400 / 348 (640: 175 /
// 167); L = 48: 116 / 180 at 128, 678 / 698 at 1536.
bool mix_token_warps(int B, int L) { return B >= (L > 16 && L <= 32 ? 768 : 1536); }

// Parts of D the mix of one token is split into (units of mix_mma_kernel): CTAs for the
// two that fit each SM, down to one 64-element step per warp (D = 4096: eight parts);
// every part sums the token's alpha again, so never more (pools of 128 / 256 tokens, L =
// 32, k = 4, D = 2048: four / three parts 85 / 116 us, two / one 73 / 93, when each part
// also read the logits of absent channels).  In the warp form so many warps that 16 fit
// each SM, down to four steps per warp (D = 4096: 16 parts).
int mix_parts(int B, int L, int D, int sms) {
  const int nc = (D / 8 + 7) / 8;
  const bool batched = mix_token_warps(B, L);
  const int most = batched ? (nc + 3) / 4 : (nc + kCoopWarps - 1) / kCoopWarps;
  const int want = batched ? (16 * sms + B - 1) / B : 2 * sms / B;
  const int parts = want < 1 ? 1 : want < most ? want : most;
  const int per = (nc + parts - 1) / parts;
  return (nc + per - 1) / per;  // no empty part
}

template <typename T>
cudaError_t launch_prenorm(const MixParams& p, cudaStream_t s) {
  const int rows = p.B * p.L;
  // as few warps to a row as hold it in registers, 1024 elements each
  auto go = [&](auto kern, int wpr) {
    const int per = kPrenormWarps / wpr;
    return launch_pdl(kern, dim3((rows + per - 1) / per), dim3(kPrenormWarps * 32), 0, s, p);
  };
  return p.D <= 1024   ? go(prenorm_kernel<T, 1>, 1)
         : p.D <= 2048 ? go(prenorm_kernel<T, 2>, 2)
                       : go(prenorm_kernel<T, 4>, 4);
}

cudaError_t launch_bf16(const MixParams& p, cudaStream_t s) {
  if (!proj_tc_supported(p)) return cudaErrorInvalidValue;  // no TMA encoder
  cudaError_t e = launch_prenorm<__nv_bfloat16>(p, s);
  if (e != cudaSuccess) return e;
  e = p.B >= kRowsTokens ? launch_router_rows(p, p.sms, s) : launch_router_tc(p, s);
  if (e != cudaSuccess) return e;
  {
    const bool warps = mix_token_warps(p.B, p.L);
    const int KS = (p.L + 15) / 16, nc = (p.D / 8 + 7) / 8;
    const int csteps = (nc + p.mix_parts - 1) / p.mix_parts;
    const size_t fr = (size_t)2 * KS * 3 * 512;
    static size_t smem_set[6][kSmemOptDevices] = {};
    const int v = KS <= 2 ? KS : 0;  // variant: layers kept in registers or not
    const size_t smem = warps ? fr * kTokenWarps : fr + (size_t)kCoopWarps * 2 * 16 * sizeof(float);
    auto kern = warps ? (v == 1   ? mix_mma_kernel<false, 1>
                         : v == 2 ? mix_mma_kernel<false, 2>
                                  : mix_mma_kernel<false, 0>)
                      : (v == 1   ? mix_mma_kernel<true, 1>
                         : v == 2 ? mix_mma_kernel<true, 2>
                                  : mix_mma_kernel<true, 0>);
    e = opt_in_smem(kern, smem, smem_set[3 * warps + v]);
    if (e != cudaSuccess) return e;
    const int units = p.B * p.mix_parts, groups = (p.k + 15) / 16;
    // Few units: their groups of 16 channels, which share nothing but the reads of h, side
    // by side, as far as two CTAs fit each SM (pools, us, one after another / so: 33 layers
    // and channels, D = 512, 3 heads of 96, 16 tokens: 42.5 / 29.3; 28, D = 264, 8 tokens:
    // 31.0 / 23.1; 128, D = 264, 2 tokens: 313 / 200; 100 tokens of 24, D = 1024: the same).
    int side = warps ? 1 : 2 * p.sms / units;
    side = side < 1 ? 1 : (side < groups ? side : groups);
    e = launch_pdl(kern, dim3(warps ? (units + kTokenWarps - 1) / kTokenWarps : units, side),
                   dim3((warps ? kTokenWarps : kCoopWarps) * 32), smem, s, p, KS, csteps);
    if (e != cudaSuccess) return e;
  }
  // tensor-core projection, QK-norm, RoPE and cache write in one kernel
  return proj_rows_supported(p) ? launch_proj_rows(p, p.sms, s) : launch_proj_tc(p, s);
}

cudaError_t launch_f32(const MixParams& p, cudaStream_t s) {
  cudaError_t e = launch_prenorm<float>(p, s);
  if (e != cudaSuccess) return e;
  {
    GemmArgs a{};
    a.W[0] = p.Wr[0];
    a.W[1] = p.Wr[1];
    a.w_stride = 0;
    a.per_branch = 1;
    a.X = p.xi;
    a.x_stride = (int64_t)p.B * p.Lp * p.D;
    a.out = p.zpart;
    a.M = p.k * p.L;
    a.N = p.B;
    a.K = p.Lp * p.D;
    a.nsplit = p.nsplit_r;
    a.k_per_split = ((a.K + p.nsplit_r - 1) / p.nsplit_r + BK - 1) / BK * BK;
    e = launch_gemm_f32(a, 2, s);
    if (e != cudaSuccess) return e;
  }
  if (p.B >= kBatchedTokens) {
    const int nvec = p.D / 8;
    const bool two = nvec > kMixThreads;  // D > 2048: two vectors per thread
    const int per = two ? (nvec + 1) / 2 : nvec;
    const int tpt = (per + 31) / 32 * 32;
    const int tb = tpt >= kMixThreads ? 1 : kMixThreads / tpt;
    const size_t per_layer = (size_t)2 * (two ? 2 : 1) * tb * tpt * 8 * sizeof(float);  // both stages
    int lc = kMixLC;
    while (lc > 1 && (size_t)lc * per_layer > kMixStageBudget) lc /= 2;
    const size_t smem = sizeof(float) * ((size_t)tb * kMixCG * p.L + (size_t)tb * p.L +
                                         (size_t)(tb * tpt / 32) * kMixCG) +
                        16 + (size_t)lc * per_layer;
    dim3 grid((p.B + tb - 1) / tb, 2, (p.k + kMixCG - 1) / kMixCG);
    auto kern = two ? mix_tokens_kernel<2> : mix_tokens_kernel<1>;
    static size_t smem_set[2][kSmemOptDevices] = {};  // per variant and device
    e = opt_in_smem(kern, smem, smem_set[two]);
    if (e != cudaSuccess) return e;
    e = launch_pdl(kern, grid, dim3(tb * tpt), smem, s, p, tpt, tb, lc);
  } else {
    const size_t smem = sizeof(float) * (kChanGroup * p.L + p.L);
    dim3 grid(p.B, 2, (p.k + kChanGroup - 1) / kChanGroup);
    e = launch_pdl(mix_kernel, grid, dim3(kMixThreads), smem, s, p);
  }
  if (e != cudaSuccess) return e;
  {
    GemmArgs a{};
    a.W[0] = p.Wkv[0];
    a.W[1] = p.Wkv[1];
    a.w_stride = (int64_t)p.Hkv * p.d * p.D;
    a.per_branch = p.k;
    a.X = p.xop;
    a.x_stride = (int64_t)p.B * p.D;
    a.out = p.proj;
    a.M = p.Hkv * p.d;
    a.N = p.B;
    a.K = p.D;
    a.nsplit = 1;
    a.k_per_split = p.D;
    e = launch_gemm_f32(a, 2 * p.k, s);
    if (e != cudaSuccess) return e;
  }
  dim3 grid(p.B, p.k, 2);
  if (p.d == 64) return launch_pdl(kv_epilogue_kernel<64>, grid, dim3(128), 0, s, p);
  if (p.d == 96) return launch_pdl(kv_epilogue_kernel<96>, grid, dim3(128), 0, s, p);
  return launch_pdl(kv_epilogue_kernel<128>, grid, dim3(128), 0, s, p);
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

MixWorkspace mix_workspace_layout(const wm_config& cfg, int32_t B, int sm_count) {
  MixWorkspace w{};
  const int Lp = (cfg.L + cfg.p - 1) / cfg.p;
  const int kL = cfg.k * cfg.L;
  const int64_t Kr = (int64_t)Lp * cfg.D;
  int ns;
  if (cfg.dtype == WM_DT_BF16) {
    ns = B >= kRowsTokens ? router_rows_splits(cfg.k, cfg.L, Lp, cfg.D, B, sm_count)
                          : router_tc_splits(cfg.k, cfg.L, Lp, cfg.D, sm_count);
  } else {
    const int tiles = 2 * ((kL + BM - 1) / BM) * ((B + BN - 1) / BN);
    ns = (2 * sm_count + tiles - 1) / tiles;
    const int max_split = (int)((Kr + 255) / 256);
    ns = ns < 1 ? 1 : (ns > max_split ? max_split : ns);
    // same rounding as the launch: whole BK blocks per split
    const int64_t kps = ((Kr + ns - 1) / ns + BK - 1) / BK * BK;
    ns = (int)((Kr + kps - 1) / kps);
  }
  w.nsplit_r = ns;
  const size_t esz = cfg.dtype == WM_DT_F32 ? 4 : 2;
  size_t off = 0;
  w.inv_rms = off; off += align256(sizeof(float) * B * cfg.L);
  w.xi = off;      off += align256(esz * 2 * (size_t)B * Kr);
  w.zpart = off;   off += align256(sizeof(float) * 2 * (size_t)ns * B * kL);
  w.rope_cs = off; off += align256(sizeof(float) * (size_t)B * cfg.d);
  w.xop = off;     off += align256(esz * 2 * (size_t)cfg.k * B * cfg.D);
  w.proj = off;    off += align256(sizeof(float) * 2 * (size_t)cfg.k * B * cfg.Hkv * cfg.d);
  w.total = off;
  return w;
}

int kv_mix_launches(const MixParams& p, int dtype) {
  if (p.B == 0) return 0;
  // prenorm, router, mix, then the tensor-core projection with its epilogue
  // or a SIMT projection and a separate epilogue
  return dtype == WM_DT_BF16 && proj_tc_supported(p) ? 4 : 5;
}

cudaError_t launch_kv_mix(MixParams& p, int dtype, int sms, cudaStream_t s) {
  p.sms = sms;
  p.mix_parts = mix_parts(p.B, p.L, p.D, sms);
  // bf16: [2][k][parts][B] floats, within the fp32 path's [2][k][B][Hkv*d] projection outputs
  if (p.mix_parts > p.Hkv * p.d) return cudaErrorInvalidConfiguration;  // (16 parts, 64 outputs)
  p.ssq = p.proj;
  return dtype == WM_DT_F32 ? launch_f32(p, s) : launch_bf16(p, s);
}

}  // namespace wm
