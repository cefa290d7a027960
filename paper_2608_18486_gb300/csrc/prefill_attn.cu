// Causal channel attention for prefill and for the token-parallel passes
// (Sec. 3.1 Step 3 "standard causal SDPA", with the dummy offset of Sec. 3.2
// and the Jacobi / cyclic Gauss-Seidel schedules of Sec. 3.3).  Query row r
// of sequence b is the query of the token at position pos[b][r]; it reads
// slots 0 .. pos of its layer's channel: the dummy and the tokens before it.
//
// Design (GB300).  A prefill pass is a dense contraction on both sides of the
// softmax, so it runs on the tcgen05 tensor cores (bf16 operands, fp32
// accumulation in TMEM), warp-specialised in the manner of flash attention on
// this architecture.  One CTA per SM (12 warps) takes work items one after
// another; an item is two 128-row query tiles of one query head, for which the
// CTA walks the 128-slot KV tiles of the sequence's channel up to each tile's
// largest position:
//    With grouped-query attention (an even number G of query heads per kv
//    head) the two tiles are the same 128 rows of two query heads that share
//    a kv head: equal causal ranges, and one K/V stream serves both.
//    Otherwise they are two consecutive 128-row tiles of one head.
//    Launches of few items (halves_pay) take one 128-row tile per item
//    instead, one half of the CTA on its even KV tiles and the other on the
//    odd ones, each with its own O, max and sum; both O lie in the same TMEM
//    lanes, so the halves merge where the rows are written.
//  * warp 8 (load): takes the next item (cluster launch control: a CTA that
//    has not started yet is cancelled and its index taken over, so the items
//    are handed out as SMs become free), publishes its rows' positions and
//    extents to the other warps, and fills Q and K through TMA (K in a ring;
//    128-byte swizzle, 64-column boxes; paged: one box per page, or per 128
//    slots of a longer page); warp 10 fills V.  (One warp for both loaded K
//    too late: it waited for V's slots, which free up half a step later.)
//    They run ahead of the other warps across items, so an item's first tiles
//    load while the last one finishes;
//  * warp 9 (MMA): S_i = Q_i K^T into TMEM, and O_i += P_i V with P_i read
//    from TMEM and V as an MN-major operand straight from its [slot][d] tile;
//    issue order PV_0(j), S_0(j+1), PV_1(j), S_1(j+1) keeps one tile's
//    matrix products running while the other tile's softmax works;
//  * warps 0-3 and 4-7 (softmax of tile 0 / 1): one thread per query row
//    reads its S row from TMEM, applies the causal mask slot <= pos (on tiles
//    the diagonal crosses), and writes the bf16 probabilities back over the S
//    columns it has read, where P V takes them as its A operand, each half as
//    it is ready.  The running max is raised, and the row of O in TMEM
//    rescaled, only when the tile's second half holds a score more than 2^8
//    above it or the first half's 64 probabilities sum to more than 2^14 (a
//    sum that is there anyway, where a max would have to be taken first).  So
//    probabilities of up to 2^14 (first half) and 2^8 (second) are used as they
//    are: fp32 sums and bf16 operands have the same relative precision
//    there, and O / l needs no correction.  They are computed with the max of the
//    tiles before, and computed again in the rare step that raises it.
// Slots beyond the item's largest position may hold anything (unwritten
// cache); their V rows are zeroed in shared memory before P V, and masked
// scores are replaced, never multiplied, so no NaN there reaches the output.
//
// What bounds it: the chain S -> softmax -> P V -> next S of each tile; with
// two tiles in turn a 128-slot step of both takes about 2900 cycles at d = 128,
// where the matrix products alone take 2048 and the 32768 exponentials 2048.
// One launch at 32 heads of 128, two prompts of 8192 positions: 939 us before
// (one item per CTA; every descriptor moved to uniform registers one by one,
// 90 cycles per MMA; 16-byte row stores at the end), 717 us now (655 replayed from a
// graph); 6/3 heads of 96, sixteen prompts of 2048: 126 and 75.5 us.
#include <limits.h>
#include <math.h>

#include "internal.h"
#include "tc.cuh"

namespace wm {
namespace {

constexpr int kPM = 128;                    // query rows per tile (MMA M)
constexpr int kPN = 128;                    // slots per KV tile
constexpr int kQT = 2;                      // query tiles per item
constexpr int kSoftWarps = 4 * kQT;         // one 4-warp group per query tile
constexpr int kLoadWarp = kSoftWarps;       // items; TMA producer of Q and K
constexpr int kMmaWarp = kSoftWarps + 1;    // MMA issuer
constexpr int kLoadVWarp = kSoftWarps + 2;  // TMA producer of V
// Three warpgroups; the last holds the load and MMA warps (its fourth warp only
// takes part in the block's barriers).  A softmax thread keeps its 128
// scores in registers, so that group hands registers over: (2 x 208 + 88) x
// 128 threads = the 384 x 168 of the launch.  (Two threads per row, 64 scores
// each, took as long per step: the 128 exponentials of a row quadrant bind.)
constexpr int kPThreads = (kSoftWarps + 4) * 32;
constexpr int kSoftRegs = 208, kIssueRegs = 88;
constexpr uint32_t kBlock = 128u * 128u;    // one 64-column block of a 128-row tile
constexpr uint32_t kTmemCols = 512;         // S_i at 128 i (P over its first 64), O_i at 256 + 128 i
constexpr double kHalvesShare = 0.4;        // see halves_pay
constexpr int kAbsent = -2;                 // position of a row past the sequence's last
constexpr float kStaleMax = 8.f;            // log2 headroom before O is rescaled
constexpr float kStaleSum = 16384.f;        // ... as a sum of 64 probabilities
constexpr uint32_t kStageBytes = 32 * 64;   // output staging of a softmax warp: 32 rows x 32 columns

template <int HD>
struct PShape {
  static constexpr int CB = (HD + 63) / 64;          // 64-column blocks of a head row
  // A slot of either ring is refilled about one and a half steps before it is
  // needed (K of step j + 2 once both S of step j are done), so two deep is
  // enough; a third K tile at d = 128 would take the output staging's place.
  static constexpr int NSK = HD <= 64 ? 4 : 2;
  static constexpr int NSV = HD <= 64 ? 4 : 2;
  static constexpr uint32_t Q_BYTES = CB * kBlock;   // one Q tile
  static constexpr uint32_t KV_BYTES = CB * kBlock;  // one K or V tile
  static constexpr uint32_t SMEM =
      kQT * Q_BYTES + (NSK + NSV) * KV_BYTES + kSoftWarps * kStageBytes + 1024;  // + alignment
  static_assert(SMEM <= 222 * 1024, "shared memory (5 KB of it static)");
};

struct PrefillParams {
  const int32_t* pos;         // [B][Tq]
  const int32_t* page_table;  // [B][max_pages]
  void* out;                  // [B][Tq][Hq][d] bf16
  int32_t* status;
  int32_t B, Tq, Hq, G, Hkv, chan, num_pages, max_pages, P, log2P;
  int32_t pair;               // 1: the two tiles are query heads 2y, 2y+1 over the same rows
  int32_t nblk, heads;        // row blocks per sequence, items' heads (or head pairs) per sequence
  int32_t group;              // (sequence, head) units walked together, see launch_prefill_attn
  float qscale;               // log2(e) / sqrt(d)
};

// One item as the load warp publishes it.
struct Item {
  int valid;       // 0: no more items
  int b, y, r0;    // sequence, head (or head pair), first row
  int nt[kQT];     // KV tiles each query tile walks
  int tmaxpos;     // largest position of the item, -1: none valid
};

// Cluster launch control: ask for the index of a CTA of this grid that has not
// started; the 16-byte answer arrives on `bar`.
__device__ __forceinline__ void clc_request(void* answer, uint64_t* bar) {
  asm volatile(
      "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(
          smem_u32(answer)),
      "r"(smem_u32(bar))
      : "memory");
}
// The answer: the CTA's x index, or -1 when none was left.
__device__ __forceinline__ int clc_answer(const void* answer) {
  uint32_t x, got;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b128 a;\n\t"
      "ld.shared.b128 a, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
      "selp.u32 %1, 1, 0, p;\n\t"
      "mov.u32 %0, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, a;\n\t}"
      : "=r"(x), "=r"(got)
      : "r"(smem_u32(answer))
      : "memory");
  return got ? (int)x : -1;
}

// max of three (one instruction on this architecture)
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// P of a KV tile for a warp in which a row has seen no score above -inf yet (m =
// -inf): zeros for such rows, and *nan_tile = s0 where they have NaN scores in the tile;
// for the others the probabilities and sums of the steps in the kernel.  S at scol is
// read again and P handed over half by half; returns the sum.  Rare, so a loop in a
// function of its own (32 heads of 128, two prompts of 8192: 672 us without it, 674 so,
// 684 as a branch of the step; as selects in the step 683 where 666 without).
__device__ __noinline__ float blank_tile(uint32_t scol, int vis, float m, float qscale, uint64_t* pfull,
                                         int lane, int* nan_tile, int s0) {
  const float nm = m == -INFINITY ? 0.f : -m;
  const float2 qs2 = make_float2(qscale, qscale), nm2 = make_float2(nm, nm);
  float2 t = make_float2(0.f, 0.f), sa = t;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    uint32_t x[32], w[16];
    tc::tmem_ld32(scol + 32 * c, x);  // (P's columns 16 c .. are read by now)
    tc::tmem_ld_wait();
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
      const float2 y = __ffma2_rn(make_float2(32 * c + e < vis ? __uint_as_float(x[e]) : -INFINITY,
                                              32 * c + e + 1 < vis ? __uint_as_float(x[e + 1]) : -INFINITY),
                                  qs2, nm2);
      const float2 pr = make_float2(ex2(y.x), ex2(y.y));
      sum = __fadd2_rn(sum, pr);
      const __nv_bfloat162 h = __floats2bfloat162_rn(pr.x, pr.y);
      w[e / 2] = m == -INFINITY ? 0u : *reinterpret_cast<const uint32_t*>(&h);
    }
    if (m == -INFINITY) {
      if (nan_tile != nullptr && !(sum.x + sum.y == 0.f)) *nan_tile = s0;
      sum = make_float2(0.f, 0.f);
    }
    tc::tmem_st16(scol + 16 * c, w);
    if ((c & 1) == 0) {
      t = sum;
      continue;
    }
    t = __fadd2_rn(t, sum);
    if (c == 1) sa = t;
    tc::tmem_st_wait();
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(&pfull[c >> 1]);
  }
  return (sa.x + t.x) + (sa.y + t.y);
}

template <int HD, bool HALVES>
__global__ void __launch_bounds__(kPThreads, 1)
    prefill_attn_kernel(const __grid_constant__ CUtensorMap tmQ,
                        const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const PrefillParams p) {
  using SH = PShape<HD>;
  constexpr int CB = SH::CB, NSK = SH::NSK, NSV = SH::NSV;
  extern __shared__ uint8_t smem_dyn[];
  __shared__ __align__(16) uint8_t clc_buf[16];
  __shared__ uint64_t clc_bar, qfull, qempty, kfull[NSK], kempty[NSK], vfull[NSV], vempty[NSV];
  // The rows past an item's last slot are zeroed in the V tile of this ring slot.  One
  // barrier per slot: its next arrival follows the slot's refill, which waits for
  // vempty, committed by the MMA thread after it has seen this one.  (One barrier for
  // all slots could be two arrivals on before the MMA thread came to its wait: the
  // tiles of two short items fit the ring.)
  __shared__ uint64_t vzero[NSV];
  __shared__ uint64_t info_full[2], info_empty[2];
  // HALVES: (max, sum) of each half's rows; xfull: a warp's are there and its O is
  // complete, xdone: it has read the other half's
  __shared__ float2 sml[HALVES ? kQT : 1][kPM];
  // A tile's NaN scores make the row NaN, unless no tile up to it had a score above -inf:
  // such a tile counts as all masked (P = 0).  Halves see every second tile, so they note
  // (first slots of) their first tile with a score above -inf and their last one of NaN
  // before it, and compare when they merge.
  __shared__ int2 sblank[HALVES ? kQT : 1][kPM];
  __shared__ uint64_t xfull[HALVES ? kQT : 1][4], xdone[HALVES ? kQT : 1][4];
  __shared__ uint64_t sfull[kQT], pfull[kQT][2], odone[kQT];  // pfull: first, second half of P
  __shared__ uint32_t tmem_base;
  __shared__ Item items[2];
  __shared__ int spos[2][kQT * kPM];        // positions of the item's rows (-1: invalid, kAbsent: past Tq)

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows_item = HALVES || p.pair ? kPM : kQT * kPM;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* Qs = base;                         // [kQT] Q tiles
  uint8_t* Ks = Qs + kQT * SH::Q_BYTES;       // [NSK] K tiles
  uint8_t* Vs = Ks + NSK * SH::KV_BYTES;      // [NSV] V tiles
  uint8_t* Os = Vs + NSV * SH::KV_BYTES;      // [kSoftWarps] output staging

  if (tid == 0) {
    mbar_init(&clc_bar, 1);
    mbar_init(&qfull, 1);
    mbar_init(&qempty, 1);
    for (int s = 0; s < NSK; ++s) {
      mbar_init(&kfull[s], 1);
      mbar_init(&kempty[s], 1);
    }
    for (int s = 0; s < NSV; ++s) {
      mbar_init(&vfull[s], 1);
      mbar_init(&vempty[s], 1);
      mbar_init(&vzero[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&info_full[i], 1);
      mbar_init(&info_empty[i], 2 + kSoftWarps);
    }
    for (int i = 0; i < kQT; ++i) {
      mbar_init(&sfull[i], 1);
      mbar_init(&pfull[i][0], 4);
      mbar_init(&pfull[i][1], 4);
      mbar_init(&odone[i], 1);
      for (int q = 0; HALVES && q < 4; ++q) {
        mbar_init(&xfull[i][q], 1);
        mbar_init(&xdone[i][q], 1);
      }
    }
    fence_mbar_init();
    tc::prefetch_tensormap(&tmQ);
    tc::prefetch_tensormap(&tmK);
    tc::prefetch_tensormap(&tmV);
  }
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, kTmemCols);
    tc::tmem_relinquish();
  }
  // programmatic dependent launch: positions, table, queries and cache may
  // come from the previous grid
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base;

  if (warp >= kSoftWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
    // Lane t of a load warp owns box t of every KV tile (one box per page, or
    // one per 128 slots of a longer page): its page id for the next tile is
    // fetched while the current tile is issued, so no page-table load sits on
    // the issue path.  Lane 0 posts the expected bytes before the lanes copy.
    const int boxes = p.P >= kPN ? 1 : kPN >> p.log2P;  // <= 16 for pages of >= 8 slots
    const int brows = p.P >= kPN ? kPN : p.P;
    // tensor-map row of this lane's box of KV tile j (-brows: read zeros)
    auto box_row = [&](int j, int b, int hkv, int tmaxpos, bool tell) -> int {
      const int s = j * kPN + lane * brows;  // first slot of the box
      const int lp = s >> p.log2P;           // logical page
      int row = -brows;
      if (lane < boxes && s <= tmaxpos && lp < p.max_pages) {
        const int pg = p.page_table[(int64_t)b * p.max_pages + lp];
        if (pg >= 0 && pg < p.num_pages)
          row = (int)((((int64_t)p.chan * p.num_pages + pg) * p.Hkv + hkv) * p.P + (s & (p.P - 1)));
        else if (tell)
          report(p.status, WM_ERR_BOUNDS);
      }
      return row;
    };
    auto load_tile = [&](const CUtensorMap* tm, uint8_t* dst, int row, uint64_t* bar) {
      if (lane == 0) mbar_arrive_expect_tx(bar, SH::KV_BYTES);
      __syncwarp();
      if (lane < boxes)
#pragma unroll
        for (int cb = 0; cb < CB; ++cb)
          tc::tma_load_2d(dst + cb * kBlock + lane * brows * 128, tm, cb * 64, row, bar);
    };
    if (warp == kLoadWarp) {
      // ============================================================== items, Q, K
      const int max_slots = p.max_pages * p.P;
      bool ok = true;
      int lin = (int)blockIdx.x;
      uint32_t kc = 0, qc = 0;  // K tiles and items' Q loaded so far
      for (uint32_t it = 0; ok; ++it) {
        const int slot = it & 1;
        if (it >= 2)
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(&info_empty[slot], ((it >> 1) - 1) & 1));
        if (!ok) break;
        if (lin < 0) {
          if (lane == 0) {
            items[slot].valid = 0;
            mbar_arrive(&info_full[slot]);
          }
          break;
        }
        // item `lin`: units of a group side by side, later rows (more work) first
        const int units = p.B * p.heads;
        const int g0 = lin / (p.group * p.nblk) * p.group;
        const int rem = lin - g0 * p.nblk, gn = min(p.group, units - g0);
        const int unit = g0 + rem % gn;
        const int b = unit / p.heads, y = unit - b * p.heads;
        const int r0 = (p.nblk - 1 - rem / gn) * rows_item;
        int mx[kQT] = {-1, -1}, ps[kQT * kPM / 32];
        bool bad = false;
#pragma unroll
        for (int u = 0; u < kQT * kPM / 32; ++u) {
          const int row = u * 32 + lane;
          ps[u] = -1;
          if (row < rows_item && r0 + row < p.Tq) ps[u] = p.pos[(int64_t)b * p.Tq + r0 + row];
        }
#pragma unroll
        for (int u = 0; u < kQT * kPM / 32; ++u) {
          const int row = u * 32 + lane;
          const bool there = row < rows_item && r0 + row < p.Tq;
          const int v = there && ps[u] >= 0 && ps[u] < max_slots ? ps[u] : -1;
          bad |= there && v < 0;
          if (row < rows_item) spos[slot][row] = there ? v : kAbsent;
          if (u < kPM / 32) mx[0] = max(mx[0], v);
          else mx[1] = max(mx[1], v);
        }
        if (bad) report(p.status, WM_ERR_BOUNDS);
        mx[0] = __reduce_max_sync(0xFFFFFFFFu, mx[0]);
        mx[1] = p.pair ? mx[0] : __reduce_max_sync(0xFFFFFFFFu, mx[1]);
        const int tmaxpos = max(mx[0], mx[1]);
        const int nmax = tmaxpos >= 0 ? tmaxpos / kPN + 1 : 0;
        if (lane == 0) {
          Item q;
          q.valid = 1;
          q.b = b;
          q.y = y;
          q.r0 = r0;
#pragma unroll
          for (int i = 0; i < kQT; ++i)
            q.nt[i] = HALVES ? (nmax + 1 - i) / 2 : mx[i] >= 0 ? mx[i] / kPN + 1 : 0;
          q.tmaxpos = tmaxpos;
          items[slot] = q;
        }
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&info_full[slot]);
          // the next item's index, needed when this item's loads are out
          mbar_arrive_expect_tx(&clc_bar, 16);
          clc_request(clc_buf, &clc_bar);
        }
        __syncwarp();
        if (nmax > 0) {
          const int hkv = (p.pair ? kQT * y : y) / p.G;  // the same kv head for both tiles
          int row_next = box_row(0, b, hkv, tmaxpos, true);
          for (int j = 0; j < nmax && ok; ++j) {
            const int row = row_next;
            if (j + 1 < nmax) row_next = box_row(j + 1, b, hkv, tmaxpos, true);
            const int sk = kc % NSK;
            if (kc >= NSK) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&kempty[sk], (kc / NSK - 1) & 1));
            if (!ok) break;
            load_tile(&tmK, Ks + sk * SH::KV_BYTES, row, &kfull[sk]);
            ++kc;
            if (j == 0) {  // the Q tiles, once every S of the last item is done with theirs
              if (qc > 0) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&qempty, (qc - 1) & 1));
              if (!ok) break;
              if (lane == 0) {
                const int nq = HALVES ? 1 : kQT;
                mbar_arrive_expect_tx(&qfull, nq * SH::Q_BYTES);
                for (int i = 0; i < nq; ++i) {
                  const int hh = p.pair ? kQT * y + i : y;
                  const int rb = p.pair ? r0 : r0 + i * kPM;
#pragma unroll
                  for (int cb = 0; cb < CB; ++cb)
                    tc::tma_load_2d(Qs + i * SH::Q_BYTES + cb * kBlock, &tmQ, hh * HD + cb * 64,
                                    b * p.Tq + rb, &qfull);
                }
              }
              __syncwarp();
              ++qc;
            }
          }
        }
        // the answer is read (or, after a failure, waited for) before its
        // buffer may be used again or given up
        const bool got = __all_sync(0xFFFFFFFFu, mbar_wait(&clc_bar, it & 1));
        ok = ok && got;
        if (!ok) break;
        lin = clc_answer(clc_buf);
        fence_proxy_async_shared();
        __syncwarp();
      }
      if (!ok && lane == 0) report(p.status, WM_ERR_TIMEOUT);
    } else if (warp == kLoadVWarp) {
      // ============================================================== V
      bool ok = true;
      uint32_t vc = 0;  // V tiles loaded so far
      for (uint32_t it = 0; ok; ++it) {
        const int slot = it & 1;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&info_full[slot], (it >> 1) & 1));
        if (!ok) break;
        const Item q = items[slot];
        __syncwarp();
        if (lane == 0) mbar_arrive(&info_empty[slot]);
        if (!q.valid) break;
        const int nmax = q.tmaxpos >= 0 ? q.tmaxpos / kPN + 1 : 0;
        if (nmax == 0) continue;
        const int hkv = (p.pair ? kQT * q.y : q.y) / p.G;
        int row_next = box_row(0, q.b, hkv, q.tmaxpos, false);  // (the K warp reports bad pages)
        for (int j = 0; j < nmax && ok; ++j) {
          const int row = row_next;
          if (j + 1 < nmax) row_next = box_row(j + 1, q.b, hkv, q.tmaxpos, false);
          const int sv = vc % NSV;
          if (vc >= NSV) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&vempty[sv], (vc / NSV - 1) & 1));
          if (!ok) break;
          load_tile(&tmV, Vs + sv * SH::KV_BYTES, row, &vfull[sv]);
          ++vc;
          const int first = q.tmaxpos - j * kPN + 1;  // slots past the largest position
          if (j + 1 == nmax && first < kPN) {
            // they may be unwritten: zero their V rows before P V reads the tile
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&vfull[sv], ((vc - 1) / NSV) & 1));
            if (!ok) break;
            uint8_t* vt = Vs + sv * SH::KV_BYTES;
            for (int r = first + lane; r < kPN; r += 32)
#pragma unroll
              for (int cb = 0; cb < CB; ++cb)
#pragma unroll
                for (int u = 0; u < 8; ++u)
                  *reinterpret_cast<uint4*>(vt + cb * kBlock + r * 128 + u * 16) =
                      make_uint4(0, 0, 0, 0);
            fence_proxy_async_shared();
            __syncwarp();
            if (lane == 0) mbar_arrive(&vzero[sv]);
          }
        }
      }
      if (!ok && lane == 0) report(p.status, WM_ERR_TIMEOUT);
    } else if (warp == kMmaWarp) {
      // ============================================================== MMA
      // One elected thread runs the schedule.  (With the whole warp in the
      // waits, each cost about 110 cycles of an idle matrix pipe, 5 a step.)
      if (tc::elect_one()) {
        const uint32_t idesc_s = tc::idesc_bf16_f32(kPM, kPN);
        const uint32_t idesc_o = tc::idesc_bf16_f32(kPM, HD) | tc::kIdescBMajorMN;
        // Descriptors of the first tiles; a tile or k-step further on adds its byte
        // offset / 16 to the address field (all of shared memory fits its 14 bits).
        const uint64_t qd0 = tc::sdesc_kmajor_sw128(smem_u32(Qs));
        const uint64_t kd0 = tc::sdesc_kmajor_sw128(smem_u32(Ks));
        const uint64_t vd0 = tc::sdesc_mnmajor_sw128(smem_u32(Vs), kBlock, 1024);
        auto issue_s = [&](int i, uint32_t st) {  // S_i = Q_i K^T, K in ring slot st
          const uint64_t qd = qd0 + (uint64_t)(HALVES ? 0u : (uint32_t)i * (SH::Q_BYTES >> 4));
          const uint64_t kd = kd0 + (uint64_t)(st * (SH::KV_BYTES >> 4));
#pragma unroll
          for (int kk = 0; kk < HD / 16; ++kk) {
            const uint64_t off = ((kk >> 2) * kBlock + (kk & 3) * 32) >> 4;
            tc::mma_bf16(tmem + 128 * i, qd + off, kd + off, idesc_s, kk > 0);
          }
          tc::mma_commit(&sfull[i]);
        };
        // O_i (+)= P_i V over half of the slots, V in ring slot st
        auto issue_pv = [&](int i, uint32_t st, bool first, int half) {
          const uint64_t vd = vd0 + (uint64_t)(st * (SH::KV_BYTES >> 4));
#pragma unroll
          for (int k2 = 0; k2 < kPN / 32; ++k2) {
            const int kk = half * (kPN / 32) + k2;
            tc::mma_bf16_ts(tmem + 256 + 128 * i, tmem + 128 * i + 8 * kk,
                            vd + (kk * 16 * 128 >> 4), idesc_o, !first || kk != 0);
          }
          if (half == 1) tc::mma_commit(&odone[i]);
        };
        bool ok = true;
        uint32_t kc = 0, vc = 0, qc = 0;  // K, V and items' Q tiles used so far
        uint32_t cnt[kQT] = {0, 0};       // P tiles used so far
        uint32_t zpar = 0;                // bit s: parity of the zeroed tiles of V slot s seen so far
        auto wait_zeroed = [&](uint32_t st) {
          const bool got = mbar_wait_spin(&vzero[st], (zpar >> st) & 1);
          zpar ^= 1u << st;
          return got;
        };
        for (uint32_t it = 0; ok; ++it) {
          const int slot = it & 1;
          ok = mbar_wait_spin(&info_full[slot], (it >> 1) & 1);
          if (!ok) break;
          const int valid = items[slot].valid, tmaxpos = items[slot].tmaxpos;
          const int nt[kQT] = {items[slot].nt[0], items[slot].nt[1]};
          mbar_arrive(&info_empty[slot]);
          if (!valid) break;
          const int nmax = tmaxpos >= 0 ? tmaxpos / kPN + 1 : 0;
          if (nmax == 0) continue;
          if constexpr (HALVES) {  // tile i: KV tiles i, i + 2, ...; each has one user
            ok = mbar_wait_spin(&qfull, qc & 1);
            if (!ok) break;
            ++qc;
            // KV tile of step j of query tile i
            auto kv_of = [&](int i, int j) -> uint32_t { return 2 * j + i; };
            auto wait_ring = [&](uint64_t* bars, uint32_t c, int ns) {
              const bool got = mbar_wait_spin(&bars[c % ns], (c / ns) & 1);
              tc::fence_after_sync();
              return got;
            };
            const bool part = tmaxpos - (nmax - 1) * kPN + 1 < kPN;  // the last V tile is zeroed in part
#pragma unroll
            for (int i = 0; i < kQT; ++i) {
              if (nt[i] == 0 || !ok) continue;
              const uint32_t c = kc + kv_of(i, 0);
              ok = wait_ring(kfull, c, NSK);
              if (!ok) continue;
              issue_s(i, c % NSK);
              tc::mma_commit(&kempty[c % NSK]);
            }
            if (!ok) break;
            if (nmax <= 2) tc::mma_commit(&qempty);
            for (int j = 0; j < nt[0]; ++j) {
#pragma unroll
              for (int i = 0; i < kQT; ++i) {
                if (j >= nt[i] || !ok) continue;
                const uint32_t kv = kv_of(i, j), st = (vc + kv) % NSV;
                ok = wait_ring(vfull, vc + kv, NSV);
                if (ok && part && kv + 1 == (uint32_t)nmax) ok = wait_zeroed(st);
                if (!ok) continue;
                ok = mbar_wait_spin(&pfull[i][0], cnt[i] & 1);
                if (!ok) continue;
                tc::fence_after_sync();
                issue_pv(i, st, j == 0, 0);
                ok = mbar_wait_spin(&pfull[i][1], cnt[i] & 1);
                if (!ok) continue;
                tc::fence_after_sync();
                issue_pv(i, st, j == 0, 1);
                ++cnt[i];
                tc::mma_commit(&vempty[st]);
                if (j + 1 < nt[i]) {
                  const uint32_t kn = kv_of(i, j + 1), c = kc + kn;
                  ok = wait_ring(kfull, c, NSK);
                  if (!ok) continue;
                  issue_s(i, c % NSK);
                  tc::mma_commit(&kempty[c % NSK]);
                  if (kn + 1 == (uint32_t)nmax) tc::mma_commit(&qempty);  // the item's last S
                }
              }
              if (!ok) break;
            }
            if (!ok) break;
            kc += nmax;
            vc += nmax;
            continue;
          }
          ok = mbar_wait_spin(&kfull[kc % NSK], (kc / NSK) & 1) && mbar_wait_spin(&qfull, qc & 1);
          if (!ok) break;
          ++qc;
          tc::fence_after_sync();
#pragma unroll
          for (int i = 0; i < kQT; ++i)
            if (nt[i] > 0) issue_s(i, kc % NSK);
          if (nmax == 1) tc::mma_commit(&qempty);
          tc::mma_commit(&kempty[kc % NSK]);
          ++kc;
          for (int j = 0; j < nmax; ++j) {
            const uint32_t st = vc % NSV;
            ok = mbar_wait_spin(&vfull[st], (vc / NSV) & 1);
            const bool more = j + 1 < nmax;
            if (ok && !more && tmaxpos - j * kPN + 1 < kPN) ok = wait_zeroed(st);
            if (!ok) break;
#pragma unroll
            for (int i = 0; i < kQT; ++i) {
              if (j >= nt[i] || !ok) continue;
              ok = mbar_wait_spin(&pfull[i][0], cnt[i] & 1);
              if (!ok) continue;
              tc::fence_after_sync();
              issue_pv(i, st, j == 0, 0);
              ok = mbar_wait_spin(&pfull[i][1], cnt[i] & 1);
              if (!ok) continue;
              tc::fence_after_sync();
              issue_pv(i, st, j == 0, 1);
              ++cnt[i];
              if (j + 1 < nt[i]) {
                ok = mbar_wait_spin(&kfull[kc % NSK], (kc / NSK) & 1);  // (at once for the second tile)
                if (!ok) continue;
                tc::fence_after_sync();
                issue_s(i, kc % NSK);
              }
            }
            if (!ok) break;
            tc::mma_commit(&vempty[st]);
            if (more) tc::mma_commit(&kempty[kc % NSK]);
            if (j + 2 == nmax) tc::mma_commit(&qempty);  // that was the item's last S
            ++vc;
            if (more) ++kc;
          }
        }
        if (!ok) report(p.status, WM_ERR_TIMEOUT);
      }
      __syncwarp();
    }
  } else {
    // ================================================================ softmax
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftRegs));
    const int i = warp >> 2, quad = warp & 3;  // query tile, TMEM lane quadrant
    const int row = quad * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t scol = lane_base + 128 * i, ocol = lane_base + 256 + 128 * i;
    uint8_t* stage = Os + warp * kStageBytes;
    uint32_t cnt = 0;  // S tiles used so far
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      const int slot = it & 1;
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(&info_full[slot], (it >> 1) & 1));
      if (!ok) break;
      const int n = items[slot].valid ? items[slot].nt[i] : -1;
      if (n < 0) break;
      // Absent rows are computed as the warp's last present one and never
      // stored: on their own masks they held every tile to the masked path.
      int mypos = spos[slot][HALVES || p.pair ? row : i * kPM + row];
      const int wpos = __reduce_max_sync(0xFFFFFFFFu, mypos);
      if (mypos == kAbsent) mypos = wpos;
      float m = -INFINITY, l = 0.f;  // max used for P (log2 units) and running sum
      if (HALVES) sblank[i][row] = make_int2(INT_MAX, -1);
      // tcgen05.ld / st are warp-collective: every lane of the warp issues each
      // one, and the wait outcomes are made warp-uniform before any branch
      for (int j = 0; j < n; ++j) {
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&sfull[i], cnt & 1));
        if (!ok) break;
        ++cnt;
        tc::fence_after_sync();
        // P goes over the S columns, slots 2c, 2c + 1 in column c
        auto hand_over = [&](int half, const uint32_t (&w)[2][16]) {
          tc::tmem_st16(scol + 32 * half, w[0]);
          tc::tmem_st16(scol + 32 * half + 16, w[1]);
          tc::tmem_st_wait();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&pfull[i][half]);
        };
        uint32_t w[2][16];
        const int s0 = (HALVES ? 2 * j + i : j) * kPN;  // the tile's first slot
        if (wpos < s0) {  // no row of the warp sees the tile (or none is present)
#pragma unroll
          for (int e = 0; e < 16; ++e) w[0][e] = w[1][e] = 0u;
          hand_over(0, w);
          hand_over(1, w);
          continue;
        }
        uint32_t v[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tc::tmem_ld32(scol + 32 * c, v[c]);
        tc::tmem_ld_wait();
        // Slots past the row's position become -inf (all 128 are visible unless
        // the diagonal crosses the tile; 32 columns at a time).
        const int vis = mypos - s0 + 1;
        if (!__all_sync(0xFFFFFFFFu, vis >= kPN)) {
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (!__all_sync(0xFFFFFFFFu, vis >= 32 * c + 32)) {
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (32 * c + e >= vis) v[c][e] = __float_as_uint(-INFINITY);
            }
        }
        // max of 64 scores (log2 units), two chains per 32 of them
        auto half_max = [&](int half) {
          float mc[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) mc[c] = -INFINITY;
#pragma unroll
          for (int e = 0; e < 16; e += 2)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int cc = 2 * half + (c >> 1), o = 16 * (c & 1) + e;
              mc[c] = max3(mc[c], __uint_as_float(v[cc][o]), __uint_as_float(v[cc][o + 1]));
            }
          // qscale > 0: the max commutes with the scale
          return fmaxf(fmaxf(mc[0], mc[1]), fmaxf(mc[2], mc[3])) * p.qscale;
        };
        // Half of P (64 slots): p = 2^(s * qscale - m) in pairs; masked slots give
        // 0 (also while the row's max is -inf).  w: packed pairs.
        float2 sum2[4];
        auto half_p = [&](int half, uint32_t (&w)[2][16]) {
          const float nm = m == -INFINITY ? 0.f : -m;
          const float2 qs2 = make_float2(p.qscale, p.qscale), nm2 = make_float2(nm, nm);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int cc = 2 * half + c;
            sum2[cc] = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              const float2 x = __ffma2_rn(
                  make_float2(__uint_as_float(v[cc][e]), __uint_as_float(v[cc][e + 1])), qs2, nm2);
              const float2 pr = make_float2(ex2(x.x), ex2(x.y));
              sum2[cc] = __fadd2_rn(sum2[cc], pr);
              const __nv_bfloat162 h = __floats2bfloat162_rn(pr.x, pr.y);
              w[c][e / 2] = *reinterpret_cast<const uint32_t*>(&h);
            }
          }
        };
        if (j == 0) {
          m = fmaxf(half_max(0), half_max(1));
          if (HALVES && m != -INFINITY) sblank[i][row].x = s0;
        }
        half_p(0, w);
        // Did the row's max grow past the headroom?  The first half's sum of
        // probabilities tells (64 of at most 2^8 each stay below 2^14, and one
        // above 2^14 shows, infinities included), the second half's max is taken
        // beside the exponentials.
        const float2 s2 = __fadd2_rn(sum2[0], sum2[1]);
        float mt1 = 0.f;
        bool raise = m == -INFINITY;
        if (!HALVES || j > 0) {  // (whole tiles were 1-2% slower with it behind the branch)
          mt1 = half_max(1);
          raise |= s2.x + s2.y > kStaleSum || mt1 > m + kStaleMax;
        }
        if (__any_sync(0xFFFFFFFFu, raise)) {
          if (j > 0) {
            // A row's max grew past the headroom: rescale O (every lane of the
            // warp takes part; rows that did not raise their max scale by 1)
            // and take the probabilities again.  P V of the previous tile is
            // in O: its MMAs were issued before the S that was waited for.
            float scale = 1.f;
            const float mt = fmaxf(half_max(0), mt1);
            raise = raise && mt > m;  // (also false while nothing is visible)
            if (raise) {
              if (HALVES && m == -INFINITY) sblank[i][row].x = s0;
              scale = ex2(m - mt);
              m = mt;
            }
            l *= scale;
#pragma unroll 1
            for (int c = 0; c < HD / 8; ++c) {
              uint32_t o[8];
              tc::tmem_ld8(ocol + 8 * c, o);
              tc::tmem_ld_wait();
#pragma unroll
              for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * scale);
              tc::tmem_st8(ocol + 8 * c, o);
            }
          }
          if (__any_sync(0xFFFFFFFFu, m == -INFINITY)) {
            l += blank_tile(scol, vis, m, p.qscale, pfull[i], lane, HALVES ? &sblank[i][row].y : nullptr, s0);
            continue;
          }
          half_p(0, w);
        }
        hand_over(0, w);
        half_p(1, w);
        hand_over(1, w);
        const float2 sa = __fadd2_rn(sum2[0], sum2[1]), sb = __fadd2_rn(sum2[2], sum2[3]);
        l += (sa.x + sb.x) + (sa.y + sb.y);
      }
      if (!ok) break;
      // ---- the item's rows: O / l, staged through shared memory so that the
      // stores cover whole sectors (a thread's own row at 16 bytes per
      // store touched 32 rows at a time: 6500-8700 cycles per item)
      if (n > 0) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&odone[i], (cnt - 1) & 1));
      if (!ok) break;
      tc::fence_after_sync();
      // Weights of this O and of the other half's.  O counts if any P V ran (else it
      // holds another item's rows) and one of its slots is visible to the row.
      bool own = n > 0 && mypos >= (HALVES ? i * kPN : 0), other = false;
      float inv = (own && l > 0.f) ? 1.f / l : 0.f, inv1 = 0.f;
      if constexpr (HALVES) {
        sml[i][row] = make_float2(m, l);
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&xfull[i][quad]);
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&xfull[i ^ 1][quad], it & 1));
        if (!ok) break;
        tc::fence_after_sync();
        const float2 o = sml[i ^ 1][row];
        const int2 mine = sblank[i][row], theirs = sblank[i ^ 1][row];
        const float mm = fmaxf(m, o.x);
        other = items[slot].nt[i ^ 1] > 0 && mypos >= (i ^ 1) * kPN;
        const float a = m != -INFINITY ? ex2(m - mm) : 0.f, b2 = o.x != -INFINITY ? ex2(o.x - mm) : 0.f;
        const float ls = a * l + b2 * o.y;
        float r = ls > 0.f ? 1.f / ls : 0.f;
        if (mine.y > theirs.x || theirs.y > mine.x) r = NAN;
        inv = a * r;
        inv1 = b2 * r;
      }
      const int b = items[slot].b, y = items[slot].y;
      const int rb = items[slot].r0 + (HALVES || p.pair ? 0 : i * kPM) + quad * 32;  // the warp's first row
      __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.out) +
                           (((int64_t)b * p.Tq + rb) * p.Hq + (p.pair ? kQT * y + i : y)) * HD;
      const int rr = lane >> 2, ch = lane & 3;  // row (of 8) and 16-byte chunk this lane stores
      const int64_t pitch = (int64_t)p.Hq * HD;
      __nv_bfloat16* drow = dst + rr * pitch + 8 * ch;
      constexpr int NC = HD / 32;
      // 32 columns of the rows: staged, and stored
      auto store_cols = [&](int c, auto x) {
#pragma unroll
        for (int e = 0; e < 32; e += 8) {
          uint32_t u[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(x(e + 2 * t), x(e + 2 * t + 1));
            u[t] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          // row `lane`, 16-byte chunk e/8, placed so that 8 rows cover all banks
          *reinterpret_cast<uint4*>(stage + lane * 64 + (((e >> 3) ^ ((lane >> 1) & 3)) << 4)) =
              make_uint4(u[0], u[1], u[2], u[3]);
        }
        __syncwarp();
        uint4 u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          u[q] = *reinterpret_cast<const uint4*>(stage + (q * 8 + rr) * 64 +
                                                 ((ch ^ ((rr >> 1) & 3)) << 4));
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (rb + q * 8 + rr < p.Tq)
            *reinterpret_cast<uint4*>(drow + q * 8 * pitch + 32 * c) = u[q];
      };
      if constexpr (HALVES) {
        // This half's share of the columns, the first one's the smaller.  Not unrolled:
        // such launches are short, a CTA runs this once or twice, and its instructions
        // are fetched meanwhile (us, unrolled / so: one prompt of 40, 12 heads of 96: 7.6 /
        // 6.8; seven of 197, 4/2 heads of 96: 8.7 / 7.4; one of 2593, 8/2 heads of 96: 24.0 /
        // 22.6; one of 40, 8 heads of 128: 7.9 / 7.0; of 64 the same).
        const int c0 = i == 1 ? NC / 2 : 0, c1 = i == 0 ? NC / 2 : NC;
#pragma unroll 1
        for (int cc = 0; cc < NC - NC / 2; ++cc) {
          const int c = c0 + cc;
          if (NC % 2 != 0 && c >= c1) break;
          uint32_t o[32], o1[32];
          tc::tmem_ld32(ocol + 32 * c, o);
          tc::tmem_ld32(lane_base + 256 + 128 * (i ^ 1) + 32 * c, o1);
          tc::tmem_ld_wait();
          store_cols(c, [&](int e) {
            return (own ? __uint_as_float(o[e]) * inv : 0.f) + (other ? __uint_as_float(o1[e]) * inv1 : 0.f);
          });
        }
      } else {
        uint32_t o[2][32];  // one group of 32 columns on its way while the last is stored
        tc::tmem_ld32(ocol, o[0]);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          tc::tmem_ld_wait();
          if (c + 1 < NC) tc::tmem_ld32(ocol + 32 * (c + 1), o[(c + 1) & 1]);
          store_cols(c, [&](int e) { return own ? __uint_as_float(o[c & 1][e]) * inv : 0.f; });
        }
      }
      tc::fence_before_sync();
      if (HALVES) {  // the next item's O and sums go over these: not before the other half has read them
        if (lane == 0) mbar_arrive(&xdone[i][quad]);
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&xdone[i ^ 1][quad], it & 1));
        if (!ok) break;
        tc::fence_after_sync();
      }
      if (lane == 0) mbar_arrive(&info_empty[slot]);  // (behind a __syncwarp of the staging)
    }
    if (!ok && lane == 0) report(p.status, WM_ERR_TIMEOUT);
  }
  // Every MMA this CTA issued has completed (each was waited on through its
  // commit barrier, or the CTA gave up after a bounded wait); release TMEM.
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
}

template <int HD, bool HALVES>
cudaError_t launch_hd(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v,
                      const PrefillParams& p, cudaStream_t s) {
  static size_t smem_set[kSmemOptDevices] = {};
  auto kern = prefill_attn_kernel<HD, HALVES>;
  if (cudaError_t e = opt_in_smem(kern, (size_t)PShape<HD>::SMEM, smem_set); e != cudaSuccess)
    return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((int64_t)p.nblk * p.heads * p.B));
  cfg.blockDim = dim3(kPThreads);
  cfg.dynamicSmemBytes = PShape<HD>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, q, k, v, p);
}

// One 128-row tile per item, its KV tiles shared out over the CTA's two halves?
// Both forms do the same steps in all; with whole tiles the launch lasts at least
// as long as its longest item (all KV tiles of the last rows), with halves half of
// that, at the price of K and V loaded once per 128 rows and head, twice as many per
// step, and of the merge.  So: where the steps of all items, causal rows evenly
// spread, fill the SMs for less than kHalvesShare of the longest item's.  Measured
// (us, whole tiles / halves; share in front): 0.11: 8 heads of 96, every eighth of
// 4575 positions 50 / 30; 0.26: 32/8 heads of 96, every eighth of 4096 48 / 36;
// 0.32: two prompts, 32/8 heads of 64, every fourth of 1000 16.5 / 12; 0.47: sixteen
// prompts, 6/3 heads of 96, every eighth of 2048 29.8 / 32.5; 0.53: two prompts of
// the 0.26 case 48.5 / 66.6 (with many CTAs the doubled K and V loads bind).  A
// sequence that has room for one KV tile only has nothing to share: one prompt of 40, 12
// heads of 64 / 96 / 128: 5.7 / 6.3 / 6.5 as whole tiles, 5.9 / 6.8 / 7.0 as halves.
bool halves_pay(const PrefillLaunch& L, int pair, int sms) {
  if ((int64_t)L.max_pages * L.P <= kPN) return false;
  const int rows_item = pair ? kPM : kQT * kPM;
  const double nblk = (L.Tq + rows_item - 1) / rows_item;
  const double items = nblk * (pair ? L.Hq / kQT : L.Hq) * L.B;
  return items * (nblk + 1) / (2 * nblk) < kHalvesShare * sms;
}

}  // namespace

cudaError_t launch_prefill_attn(const PrefillLaunch& L, int sms, cudaStream_t s) {
  CUtensorMap tq, tk, tv;
  const uint64_t pool_rows = (uint64_t)L.k * L.num_pages * L.Hkv * L.P;
  const uint32_t box_rows = L.P >= kPN ? (uint32_t)kPN : (uint32_t)L.P;
  if (!tma_map_bf16_2d(&tq, L.q, (uint64_t)L.B * L.Tq, (uint64_t)L.Hq * L.d,
                       (uint64_t)L.Hq * L.d, (uint32_t)kPM) ||
      !tma_map_bf16_2d(&tk, L.k_pool, pool_rows, L.d, L.d, box_rows) ||
      !tma_map_bf16_2d(&tv, L.v_pool, pool_rows, L.d, L.d, box_rows))
    return cudaErrorInvalidValue;
  PrefillParams p{};
  p.pos = L.pos;
  p.page_table = L.page_table;
  p.out = L.out;
  p.status = L.status;
  p.B = L.B;
  p.Tq = L.Tq;
  p.Hq = L.Hq;
  p.G = L.Hq / L.Hkv;
  p.pair = (p.G % kQT == 0) ? 1 : 0;
  p.Hkv = L.Hkv;
  p.chan = L.chan;
  p.num_pages = L.num_pages;
  p.max_pages = L.max_pages;
  p.P = L.P;
  int lg = 0;
  while ((1 << lg) < L.P) ++lg;
  p.log2P = lg;
  const bool halves = halves_pay(L, p.pair, sms);
  if (halves) p.pair = 0;
  const int rows_item = halves || p.pair ? kPM : kQT * kPM;
  p.nblk = (L.Tq + rows_item - 1) / rows_item;
  p.heads = p.pair ? L.Hq / kQT : L.Hq;
  if ((int64_t)p.nblk * p.heads * L.B > INT32_MAX) return cudaErrorInvalidConfiguration;
  // Items run in the order of their index: within a group of (sequence, head)
  // units all last row blocks first, so that the launch ends with short items;
  // a group's K and V (64 MB at most) stay in L2 while its row blocks pass.
  const int64_t kv_bytes = (int64_t)L.max_pages * L.P * L.d * 4;
  const int64_t fit = (64ll << 20) / kv_bytes, units = (int64_t)p.heads * L.B;
  const int64_t groups = fit < 1 ? units : (units + fit - 1) / fit;  // of near-equal size
  p.group = (int)((units + groups - 1) / groups);
  p.qscale = (float)(1.4426950408889634 / sqrt((double)L.d));
  switch (L.d) {
    case 64: return halves ? launch_hd<64, true>(tq, tk, tv, p, s) : launch_hd<64, false>(tq, tk, tv, p, s);
    case 96: return halves ? launch_hd<96, true>(tq, tk, tv, p, s) : launch_hd<96, false>(tq, tk, tv, p, s);
    case 128: return halves ? launch_hd<128, true>(tq, tk, tv, p, s) : launch_hd<128, false>(tq, tk, tv, p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace wm
