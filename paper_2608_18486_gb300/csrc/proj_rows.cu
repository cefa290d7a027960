// The pool's two dense contractions for groups of tokens (prefill, the token-
// parallel passes of Sec. 3.3) on the tcgen05 tensor cores: bf16 operands, fp32
// accumulation in TMEM.
//  * projection (Sec. 3.1 Step 2): K_j = W^K_j x^K_j, V_j = W^V_j x^V_j, then
//    per-head QK-norm and RoPE on keys, bf16 rounding and the write to each
//    token's cache slot;
//  * router logits W^alpha xi (Sec. 3.1 Step 1), split over the L'D reduction,
//    each split storing fp32 partial sums.
//
// Shape: with hundreds of tokens the tokens take the MMA's M side (128 of them),
// the weight rows its N side, so an epilogue thread owns one token: the norm
// over a head is a sum over its own registers and RoPE needs no exchange.
// (proj_tc.cu, for decode steps, has the weights on M; with 4096 tokens its
// epilogue, a warp per (token, head) through shared memory and not overlapped
// with the next tile, took most of 196 us at D = 512, 3 heads of 96, k = 16.)
//
// Persistent CTAs, one per SM; each walks a contiguous run of tiles.  A tile is
// 128 tokens of one branch and channel against up to U units of SW weight rows
// (whole heads).  Every unit accumulates in its own TMEM slot (NSLOT of them in
// a ring), so the next tile's MMAs run while this one's units are drained:
//  * warp 0: TMA of activation and weight k-blocks (64 columns, 128-byte
//    swizzle) through an mbarrier ring;
//  * warp 1: MMAs, from one elected thread;
//  * (warps 2-3 only hand over their registers;)
//  * warps 4-11: epilogue, two groups of four (one TMEM lane quadrant each)
//    taking turns at the units; a unit's slot is free again once it is in
//    registers.  They also load the RoPE table of the tile's tokens, transposed
//    to [pair][token] (by two warps alone that took 20 us).  Outputs go through a small staging buffer so that a store
//    covers whole 64-byte runs of the scattered cache rows.
// Tiles run token tile by token tile, so the table is loaded once or twice per
// CTA and the activations of a tile are read once; the weights (9 MB there) come
// from L2.  Measured: 58 us for the projection (196 before), 23 us for the
// router (47 before) at 4096 tokens of that shape.
#include <math.h>

#include "internal.h"
#include "tc.cuh"

namespace wm {
namespace {

constexpr int kRM = 128;                   // tokens per tile (MMA M)
constexpr int kRBK = 64;                   // K elements per stage (128 bytes of bf16)
constexpr int kRStages = 3;
constexpr int kEpiWarp0 = 4, kEpiWarps = 8;
constexpr int kRThreads = (kEpiWarp0 + kEpiWarps) * 32;
// An epilogue thread holds a head in registers (128 of them at d = 128): the first
// warpgroup hands over, (2 x 208 + 88) x 128 threads = the 384 x 168 of the launch.
constexpr int kEpiRegs = 208, kIssueRegs = 88;
constexpr uint32_t kRStage = 32 * 64;      // staging of an epilogue warp: 32 rows x 64 bytes

enum { kRowsKV = 0, kRowsPartial = 1 };

template <int HD>
struct RShape {
  static constexpr int SW = HD == 64 ? 128 : HD;   // weight rows per unit (MMA N)
  static constexpr int HPU = SW / HD;              // heads per unit
  static constexpr int U = HD == 96 ? 3 : 2;       // units per tile
  static constexpr int NSLOT = 512 / SW;           // TMEM slots
  static constexpr uint32_t A_BYTES = kRM * 128;
  static constexpr uint32_t W_BYTES = SW * 128;    // one unit
  static constexpr uint32_t TAB = kRM * (HD / 2) * 8;
  static constexpr uint32_t SMEM =
      kRStages * (A_BYTES + U * W_BYTES) + TAB + kEpiWarps * kRStage + 1024;
  static_assert(SMEM <= 226 * 1024, "shared memory");
};

struct RowsParams {
  int32_t B, k, Hkv, M_item;      // tokens, channels; weight rows per channel
  int32_t nunits, nn;             // units per channel, tiles per (channel, token tile)
  int32_t nk, kb_per_split, nsplit, M_total;  // k-blocks; router: per split, splits, rows of W
  int32_t tiles;
  float* zpart;                   // router: [2][nsplit][B][M_total]
  int32_t P, log2P, num_pages, max_pages, parts;
  float eps_qk, eps_rms, inv_D;
  const int32_t* page_table;
  const int32_t* slot;
  __nv_bfloat16* k_pool;
  __nv_bfloat16* v_pool;
  const __nv_bfloat16* qk_g;
  const float* rope_cs;
  const float* ssq;               // [2][k][parts][B] sums of squares of the operand
  int32_t* status;
};

// A tile: token tile tt, branch X, channel (projection) or split (router) j,
// units n*U .. of it.  n runs fastest, then j, X, tt.
struct Tile {
  int tt, X, j, n;
};
__device__ __forceinline__ Tile tile_of(int x, int nn, int nj) {
  Tile t;
  t.n = x % nn;
  x /= nn;
  t.j = x % nj;
  x /= nj;
  t.X = x & 1;
  t.tt = x >> 1;
  return t;
}

template <int HD, int MODE>
__global__ void __launch_bounds__(kRThreads, 1)
    proj_rows_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                     const __grid_constant__ CUtensorMap tmX, const RowsParams p) {
  using SH = RShape<HD>;
  constexpr int SW = SH::SW, U = SH::U, NSLOT = SH::NSLOT, HALF = HD / 2, NS = kRStages;
  extern __shared__ uint8_t smem_dyn[];
  __shared__ uint64_t full[NS], empty[NS], sfull[NSLOT], sempty[NSLOT], tfull, tempty;
  __shared__ uint32_t tmem_base;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* As = base;                                     // [NS]
  uint8_t* Ws = As + NS * SH::A_BYTES;                    // [NS][U]
  float2* tab = reinterpret_cast<float2*>(Ws + NS * U * SH::W_BYTES);  // [HALF][kRM] (cos, sin)
  uint8_t* stage0 = reinterpret_cast<uint8_t*>(tab) + SH::TAB;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nj = MODE == kRowsKV ? p.k : p.nsplit;
  const int x0 = (int)((int64_t)blockIdx.x * p.tiles / gridDim.x);
  const int x1 = (int)((int64_t)(blockIdx.x + 1) * p.tiles / gridDim.x);
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < NSLOT; ++s) {
      mbar_init(&sfull[s], 1);
      mbar_init(&sempty[s], 4);
    }
    mbar_init(&tfull, kEpiWarps);
    mbar_init(&tempty, kEpiWarps);
    fence_mbar_init();
    tc::prefetch_tensormap(&tmW0);
    tc::prefetch_tensormap(&tmW1);
    tc::prefetch_tensormap(&tmX);
  }
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, 512);
    tc::tmem_relinquish();
  }
  // programmatic dependent launch: the activations come from the previous grid
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;

  // k-blocks of a tile
  auto kb_range = [&](const Tile& t, int& kb0, int& kb1) {
    kb0 = MODE == kRowsKV ? 0 : t.j * p.kb_per_split;
    kb1 = MODE == kRowsKV ? p.nk : min(p.nk, kb0 + p.kb_per_split);
  };

  if (warp < kEpiWarp0) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
  if (warp == 0) {
    if (tc::elect_one()) {
      // ============================================================ TMA
      bool ok = true;
      uint32_t c = 0;  // stages filled
      for (int x = x0; x < x1 && ok; ++x) {
        const Tile t = tile_of(x, p.nn, nj);
        const int nu = min(U, p.nunits - t.n * U);
        const int xrow = (MODE == kRowsKV ? (t.X * p.k + t.j) * p.B : t.X * p.B) + t.tt * kRM;
        const int wrow = (MODE == kRowsKV ? t.j * p.M_item : 0) + t.n * U * SW;
        int kb0, kb1;
        kb_range(t, kb0, kb1);
        for (int kb = kb0; kb < kb1; ++kb, ++c) {
          const uint32_t s = c % NS;
          if (c >= NS) ok = mbar_wait(&empty[s], (c / NS - 1) & 1);
          if (!ok) break;
          mbar_arrive_expect_tx(&full[s], SH::A_BYTES + nu * SH::W_BYTES);
          tc::tma_load_2d(As + s * SH::A_BYTES, &tmX, kb * kRBK, xrow, &full[s]);
          for (int u = 0; u < nu; ++u)
            tc::tma_load_2d(Ws + (s * U + u) * SH::W_BYTES, t.X == 0 ? &tmW0 : &tmW1, kb * kRBK,
                            wrow + u * SW, &full[s]);
        }
      }
      if (!ok) report(p.status, WM_ERR_TIMEOUT);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (tc::elect_one()) {
      // ============================================================ MMA
      const uint32_t idesc = tc::idesc_bf16_f32(kRM, SW);
      const uint64_t ad0 = tc::sdesc_kmajor_sw128(smem_u32(As));
      const uint64_t wd0 = tc::sdesc_kmajor_sw128(smem_u32(Ws));
      bool ok = true;
      uint32_t c = 0, uc = 0;  // stages, units used
      for (int x = x0; x < x1 && ok; ++x) {
        const Tile t = tile_of(x, p.nn, nj);
        const int nu = min(U, p.nunits - t.n * U);
        int kb0, kb1;
        kb_range(t, kb0, kb1);
        for (int u = 0; u < nu && ok; ++u) {
          const uint32_t q = uc + u;
          if (q >= NSLOT) ok = mbar_wait_spin(&sempty[q % NSLOT], (q / NSLOT - 1) & 1);
        }
        if (!ok) break;
        tc::fence_after_sync();
        for (int kb = kb0; kb < kb1; ++kb, ++c) {
          const uint32_t s = c % NS;
          ok = mbar_wait_spin(&full[s], (c / NS) & 1);
          if (!ok) break;
          tc::fence_after_sync();
          const uint64_t ad = ad0 + s * (SH::A_BYTES >> 4);
          const uint64_t wd = wd0 + s * (U * SH::W_BYTES >> 4);
#pragma unroll
          for (int kk = 0; kk < kRBK / 16; ++kk)
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (u < nu)
                tc::mma_bf16(tmem + ((uc + u) % NSLOT) * SW, ad + kk * 2,
                             wd + u * (SH::W_BYTES >> 4) + kk * 2, idesc, kb > kb0 || kk > 0);
          tc::mma_commit(&empty[s]);
        }
        if (!ok) break;
        for (int u = 0; u < nu; ++u) tc::mma_commit(&sfull[(uc + u) % NSLOT]);
        uc += nu;
      }
      if (!ok) report(p.status, WM_ERR_TIMEOUT);
    }
    __syncwarp();
  }
  } else {
    // ================================================================ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    const int grp = (warp - kEpiWarp0) >> 2, quad = warp & 3;
    const int row = quad * 32 + lane;  // this thread's token of the tile
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    uint8_t* stage = stage0 + (warp - kEpiWarp0) * kRStage;
    const int sr = lane >> 2, sc = lane & 3;  // row (of 8) and 16-byte chunk this lane stores
    uint8_t* put = stage + lane * 64;         // chunk c of this thread's row goes to put + swz(c)
    auto swz = [&](int r, int c) { return (c ^ ((r >> 1) & 3)) << 4; };
    int last = -1;
    uint32_t nt = 0, uc = 0;
    bool ok = true;
    int64_t ro[4];  // cache row of the four token rows this lane stores, -1: none
    for (int x = x0; x < x1 && ok; ++x) {
      const Tile t = tile_of(x, p.nn, nj);
      const int nu = min(U, p.nunits - t.n * U);
      if (t.tt != last) {
        if (MODE == kRowsKV && last >= 0) {  // every warp is done with the old table
          __syncwarp();
          if (lane == 0) mbar_arrive(&tempty);
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tempty, (nt - 1) & 1));
          if (!ok) break;
        }
        last = t.tt;
        if (MODE == kRowsKV) {
          const int tok = t.tt * kRM + row;
          int64_t mine = -1;
          if (tok < p.B) {
            const int s = p.slot[tok];
            int pg = -1;
            if (s >= 1 && s < p.max_pages * p.P)
              pg = p.page_table[(int64_t)tok * p.max_pages + (s >> p.log2P)];
            if (pg >= 0 && pg < p.num_pages)
              mine = (int64_t)pg * p.Hkv * p.P + (s & (p.P - 1));
            else
              report(p.status, WM_ERR_BOUNDS);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) ro[q] = __shfl_sync(0xFFFFFFFFu, mine, q * 8 + sr);
          // this thread's token, every other pair of pairs: 16-byte loads, all in
          // flight, conflict-free stores
          if (tok < p.B) {
            const float4* src = reinterpret_cast<const float4*>(p.rope_cs + (int64_t)tok * HD);
#pragma unroll
            for (int i = 0; i < HALF / 4; ++i) {
              const float4 f = src[2 * i + grp];
              tab[(4 * i + 2 * grp) * kRM + row] = make_float2(f.x, f.y);
              tab[(4 * i + 2 * grp + 1) * kRM + row] = make_float2(f.z, f.w);
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&tfull);
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tfull, nt & 1));
          ++nt;
          if (!ok) break;
        }
      }
      float scale = 0.f;  // 1/RMS of channel j's state
      if (MODE == kRowsKV) {
        const int tok = min(t.tt * kRM + row, p.B - 1);
        const float* sq = p.ssq + (int64_t)(t.X * p.k + t.j) * p.parts * p.B + tok;
        for (int q = 0; q < p.parts; ++q) scale += sq[(int64_t)q * p.B];
        scale = rsqrtf(scale * p.inv_D + p.eps_rms);
      }
      for (int u = 0; u < nu && ok; ++u, ++uc) {
        if ((int)(uc & 1) != grp) continue;
        const uint32_t slot = uc % NSLOT;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&sfull[slot], (uc / NSLOT) & 1));
        if (!ok) break;
        tc::fence_after_sync();
#pragma unroll
        for (int hl = 0; hl < SH::HPU; ++hl) {
          uint32_t y[HD / 32][32];
#pragma unroll
          for (int c = 0; c < HD / 32; ++c)
            tc::tmem_ld32(lane_base + slot * SW + hl * HD + 32 * c, y[c]);
          tc::tmem_ld_wait();
          if (hl == SH::HPU - 1) {  // the unit is in registers: its slot may be written again
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sempty[slot]);
          }
          auto f = [&](int i) { return __uint_as_float(y[i >> 5][i & 31]); };
          if (MODE == kRowsPartial) {
            // zpart[X][split][token][m0 ..], 16 columns at a time
            const int m0 = (t.n * U + u) * SW;
            float* z = p.zpart + (((int64_t)t.X * p.nsplit + t.j) * p.B + t.tt * kRM + quad * 32) * p.M_total;
#pragma unroll
            for (int c0 = 0; c0 < HD; c0 += 16) {
              if (m0 + c0 >= p.M_total) break;
#pragma unroll
              for (int c = 0; c < 4; ++c)
                *reinterpret_cast<float4*>(put + swz(lane, c)) =
                    make_float4(f(c0 + 4 * c), f(c0 + 4 * c + 1), f(c0 + 4 * c + 2), f(c0 + 4 * c + 3));
              __syncwarp();
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int r = q * 8 + sr, m = m0 + c0 + 4 * sc;
                const float4 v = *reinterpret_cast<const float4*>(stage + r * 64 + swz(r, sc));
                if (t.tt * kRM + quad * 32 + r >= p.B) continue;
                float* d = z + (int64_t)r * p.M_total + m;
                if ((p.M_total & 3) == 0) {
                  if (m < p.M_total) *reinterpret_cast<float4*>(d) = v;
                } else {
                  if (m < p.M_total) d[0] = v.x;
                  if (m + 1 < p.M_total) d[1] = v.y;
                  if (m + 2 < p.M_total) d[2] = v.z;
                  if (m + 3 < p.M_total) d[3] = v.w;
                }
              }
              __syncwarp();
            }
            continue;
          }
          const int hh = (t.n * U + u) * SH::HPU + hl;
          if (hh >= p.Hkv) continue;  // (warp-uniform) rows past the last head
          __nv_bfloat16* pool = (t.X == 0 ? p.k_pool : p.v_pool) +
                                ((int64_t)t.j * p.num_pages * p.Hkv * p.P + (int64_t)hh * p.P) * HD;
          float k1 = scale;
          if (t.X == 0) {  // QK-norm over the head, of the scaled projection
            float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int i = 0; i < HD; ++i) {
              const float v = f(i) * scale;
              s4[i & 3] = fmaf(v, v, s4[i & 3]);
            }
            k1 *= rsqrtf(((s4[0] + s4[1]) + (s4[2] + s4[3])) / (float)HD + p.eps_qk);
          }
          const __nv_bfloat16* qg = p.qk_g + (int64_t)t.j * HD;
          // 16 elements of each half of the row at a time (one 64-byte staging row)
#pragma unroll
          for (int i0 = 0; i0 < HALF; i0 += 16) {
            uint32_t o[2][8];
#pragma unroll
            for (int e8 = 0; e8 < 16; e8 += 8) {
              float g0[8], g1[8];
              if (t.X == 0) {
                Elem<__nv_bfloat16>::unpack(__ldg(reinterpret_cast<const uint4*>(qg + i0 + e8)), g0);
                Elem<__nv_bfloat16>::unpack(__ldg(reinterpret_cast<const uint4*>(qg + HALF + i0 + e8)), g1);
              }
#pragma unroll
              for (int e = 0; e < 8; e += 2) {
                float a[2], c[2];
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                  const int i = i0 + e8 + e + w;
                  a[w] = f(i) * k1;
                  c[w] = f(i + HALF) * k1;
                  if (t.X == 0) {  // gain, then rotate-half RoPE
                    const float2 cs = tab[i * kRM + row];
                    const float x0 = a[w] * g0[e + w], x1 = c[w] * g1[e + w];
                    a[w] = x0 * cs.x - x1 * cs.y;
                    c[w] = x1 * cs.x + x0 * cs.y;
                  }
                }
                const __nv_bfloat162 ha = __floats2bfloat162_rn(a[0], a[1]);
                const __nv_bfloat162 hc = __floats2bfloat162_rn(c[0], c[1]);
                o[0][(e8 + e) / 2] = *reinterpret_cast<const uint32_t*>(&ha);
                o[1][(e8 + e) / 2] = *reinterpret_cast<const uint32_t*>(&hc);
              }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)  // chunks 0, 1: first half of the row; 2, 3: second
              *reinterpret_cast<uint4*>(put + swz(lane, c)) =
                  make_uint4(o[c >> 1][4 * (c & 1)], o[c >> 1][4 * (c & 1) + 1],
                             o[c >> 1][4 * (c & 1) + 2], o[c >> 1][4 * (c & 1) + 3]);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int r = q * 8 + sr;
              const uint4 v = *reinterpret_cast<const uint4*>(stage + r * 64 + swz(r, sc));
              if (ro[q] >= 0)
                *reinterpret_cast<uint4*>(pool + ro[q] * HD + (sc >> 1) * HALF + i0 + 8 * (sc & 1)) = v;
            }
            __syncwarp();
          }
        }
      }
    }
    if (!ok && lane == 0) report(p.status, WM_ERR_TIMEOUT);
  }
  // Every MMA has completed (its unit was waited for through its commit, or a
  // bounded wait gave up); release TMEM.
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 512);
  }
}

template <int HD, int MODE>
cudaError_t launch_rows(const CUtensorMap& w0, const CUtensorMap& w1, const CUtensorMap& x,
                        const RowsParams& p, int sms, cudaStream_t s) {
  static size_t smem_set[kSmemOptDevices] = {};
  auto kern = proj_rows_kernel<HD, MODE>;
  if (cudaError_t e = opt_in_smem(kern, (size_t)RShape<HD>::SMEM, smem_set); e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.tiles < sms ? p.tiles : sms));
  cfg.blockDim = dim3(kRThreads);
  cfg.dynamicSmemBytes = RShape<HD>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, w0, w1, x, p);
}

template <int HD>
cudaError_t launch_kv(const MixParams& mp, int sms, cudaStream_t s) {
  using SH = RShape<HD>;
  RowsParams p{};
  p.B = mp.B;
  p.k = mp.k;
  p.Hkv = mp.Hkv;
  p.M_item = mp.Hkv * HD;
  p.nunits = (p.M_item + SH::SW - 1) / SH::SW;
  p.nn = (p.nunits + SH::U - 1) / SH::U;
  p.nk = (mp.D + kRBK - 1) / kRBK;
  p.tiles = (mp.B + kRM - 1) / kRM * 2 * mp.k * p.nn;
  p.P = mp.P;
  p.log2P = mp.log2P;
  p.num_pages = mp.num_pages;
  p.max_pages = mp.max_pages;
  p.parts = mp.mix_parts;
  p.eps_qk = mp.eps_qk;
  p.eps_rms = mp.eps_rms;
  p.inv_D = 1.f / (float)mp.D;
  p.page_table = mp.page_table;
  p.slot = mp.slot;
  p.k_pool = reinterpret_cast<__nv_bfloat16*>(mp.k_pool);
  p.v_pool = reinterpret_cast<__nv_bfloat16*>(mp.v_pool);
  p.qk_g = reinterpret_cast<const __nv_bfloat16*>(mp.qk_g);
  p.rope_cs = mp.rope_cs;
  p.ssq = mp.ssq;
  p.status = mp.status;
  CUtensorMap tw[2], tx;
  for (int X = 0; X < 2; ++X)
    if (!tma_map_bf16_2d(&tw[X], mp.Wkv[X], (uint64_t)mp.k * p.M_item, mp.D, mp.D, SH::SW))
      return cudaErrorInvalidValue;
  if (!tma_map_bf16_2d(&tx, mp.xop, (uint64_t)2 * mp.k * mp.B, mp.D, mp.D, kRM))
    return cudaErrorInvalidValue;
  return launch_rows<HD, kRowsKV>(tw[0], tw[1], tx, p, sms, s);
}

}  // namespace

// From kRowsTokens (128: a whole tile) on the pool's contractions take the tokens as
// MMA rows: below, the decode form (proj_tc.cu) pads fewer rows of its 16-token
// granularity, above, its accumulators and epilogue grow with the tokens of a CTA.
// Whole pools (us, decode form / this one) at 64, 96, 128 and 256 tokens: L = k = 16, D =
// 512, 3 heads of 96: 23.0 / 25.2, 25.7 / 25.7, 29.3 / 28.6, 39.0 / 30.1; L = k = 16, D =
// 1024, 8 heads of 128: 32.0 / 34.0, 37.9 / 36.5, 62.5 / 39.6, 76.6 / 51.7; L = 32, k =
// 4, D = 2048, 8 heads of 128: 40.7 / 43.2, 50.6 / 51.5, 57.6 / 56.4, 90.0 / 77.7 (160:
// 67.0 / 69.2); L = 32, k = 16, D = 4096, 32 heads of 128: 239 / 250, 281 / 267, 361 /
// 287, 563 / 408.
bool proj_rows_supported(const MixParams& mp) {
  return mp.B >= kRowsTokens && (reinterpret_cast<uintptr_t>(mp.qk_g) % 16) == 0;
}

// Router splits over the reduction: as many as leave every tile its own SM.
int router_rows_splits(int k, int L, int Lp, int D, int B, int sms) {
  const int nk = (Lp * D + kRBK - 1) / kRBK;
  const int tiles = (B + kRM - 1) / kRM * 2 * ((k * L + 255) / 256);
  int ns = sms / tiles;
  const int max_ns = nk / 8 > 1 ? nk / 8 : 1;  // at least 8 k-blocks per split
  ns = ns < 1 ? 1 : (ns > max_ns ? max_ns : ns);
  const int per = (nk + ns - 1) / ns;
  return (nk + per - 1) / per;
}

cudaError_t launch_proj_rows(const MixParams& mp, int sms, cudaStream_t s) {
  if (mp.d == 64) return launch_kv<64>(mp, sms, s);
  if (mp.d == 96) return launch_kv<96>(mp, sms, s);
  return launch_kv<128>(mp, sms, s);
}

cudaError_t launch_router_rows(const MixParams& mp, int sms, cudaStream_t s) {
  using SH = RShape<128>;
  const int kL = mp.k * mp.L, K = mp.Lp * mp.D;
  RowsParams p{};
  p.B = mp.B;
  p.k = mp.k;
  p.nunits = (kL + SH::SW - 1) / SH::SW;
  p.nn = (p.nunits + SH::U - 1) / SH::U;
  p.nk = (K + kRBK - 1) / kRBK;
  p.nsplit = mp.nsplit_r;
  p.kb_per_split = (p.nk + mp.nsplit_r - 1) / mp.nsplit_r;
  p.M_total = kL;
  p.zpart = mp.zpart;
  p.tiles = (mp.B + kRM - 1) / kRM * 2 * p.nsplit * p.nn;
  p.status = mp.status;
  CUtensorMap tw[2], tx;
  for (int X = 0; X < 2; ++X)
    if (!tma_map_bf16_2d(&tw[X], mp.Wr[X], (uint64_t)kL, K, K, SH::SW)) return cudaErrorInvalidValue;
  if (!tma_map_bf16_2d(&tx, mp.xi, (uint64_t)2 * mp.B, K, K, kRM)) return cudaErrorInvalidValue;
  return launch_rows<128, kRowsPartial>(tw[0], tw[1], tx, p, sms, s);
}

}  // namespace wm
