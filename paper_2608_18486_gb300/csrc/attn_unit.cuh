#pragma once
// Decode attention over one channel of the paged k-channel cache, unit split
// (Sec. 3.1 Step 3; dummy slot of Sec. 3.2), for launches with few
// (sequence b, kv head h) units: the paper's own model shape (16 sequences x
// 3 kv heads) has 48 of them for 152 SMs.
//
// Design.  Each unit gets one thread-block cluster of C CTAs (at most 8, all
// clusters resident at once), and each of its C x NW warps streams a contiguous,
// near-equal share of the unit's stages through a private 3-deep ring of bulk
// async copies, with the same stage math as the stream-K kernel
// (attn_kernel.cuh).  The partial softmax states then merge on chip: the
// warps of a CTA through shared memory, the CTAs of the cluster through
// distributed shared memory, each CTA producing 1/C of the unit's G x d
// outputs.  No record goes through global memory and no flag or ticket is
// waited on; the stream-K kernel's cross-SM merge (flags raised on other SMs,
// records landed from L2) sits on the critical path of such short launches.
// The split is static, so it suits launches whose units have similar lengths;
// the planner takes it for launches below 2 GB, or of one sequence, when all
// its clusters are resident at once with enough warps (csrc/wm_api.cu).
#include <cooperative_groups.h>

#include "attn_kernel.cuh"

namespace wm {
namespace attn_unit_detail {

namespace cg = cooperative_groups;
using attn_detail::CopyShape;
using attn_detail::kDtype;
using attn_detail::MathPick;
using attn_detail::Shape;

constexpr int kUStages = 3;  // ring depth per warp

// Warps per CTA: 4 where a kv head has at most two query heads (two or
// three CTAs per SM, by the stage size: smaller CTAs keep more clusters
// resident and more SMs busy), else 8 (one CTA per SM: fp32 states of four or
// eight query heads take up to 255 registers, and few units need the warps), or
// 4 if the planner asks for them (bf16: more units than SMs).
constexpr int unit_warps(int G) { return G <= 2 ? 4 : 8; }
// CTAs per SM the register budget is sized for (at most 12 warps of 170
// registers per SM; the stages of four or eight heads of 64 or 128 leave room for 8)
constexpr int unit_min_blocks(int nw, int g, int d) { return nw > 4 ? 1 : g > 2 && d != 96 ? 2 : 3; }

// floats of one partial state: G x HD unnormalised outputs, then (max, sum)
// per query head (log2 units)
constexpr int unit_rec(int G, int HD) { return G * HD + 2 * G; }

// MMA: stage math on the tensor cores (attn_unit_mma)
template <typename T, int HD, int G, int SB, int NW, bool MMA>
__global__ void __launch_bounds__(NW * 32, unit_min_blocks(NW, G, HD)) decode_attn_unit_kernel(const AttnParams p) {
  using SH = Shape<T, HD, SB>;
  using MATH = typename MathPick<T, HD, G, SB, MMA>::type;
  constexpr int STAGE_SLOTS = SH::STAGE_SLOTS;
  constexpr int K_ELEMS = SH::STAGE_ELEMS;             // of K in the ring
  constexpr int RING_ELEMS = 2 * K_ELEMS + MATH::kPad;  // of K and V
  constexpr uint32_t KV_BYTES = K_ELEMS * sizeof(T);
  constexpr int E = G * HD;  // output elements of a unit
  constexpr int REC = unit_rec(G, HD);
  constexpr unsigned FULLMASK = 0xFFFFFFFFu;
  // a warp's state goes into its own ring once the ring is idle
  static_assert((size_t)REC * sizeof(float) <= (size_t)kUStages * 2 * KV_BYTES, "record fits the ring");

  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);  // [NW][S][RING_ELEMS]
  float* crec = reinterpret_cast<float*>(ring + NW * kUStages * RING_ELEMS);  // [REC]
  __shared__ uint64_t bars[NW][kUStages];
  __shared__ uint64_t masks[NW][kUStages];

  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int rank = (int)cluster.block_rank();
  const int unit = (int)(blockIdx.x / (unsigned)C);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = unit / p.Hkv, h = unit - b * p.Hkv;
  const int max_slots = p.max_pages * p.P;

  // Programmatic dependent launch, as in the stream-K kernel: with the
  // caller's inputs_ready promise the cache, table and lengths are read
  // before the dependency wait, and only the query after it.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const bool early = p.inputs_ready != 0;
  if (!early) asm volatile("griddepcontrol.wait;" ::: "memory");

  if (tid == 0) {
    for (int w = 0; w < NW; ++w)
      for (int s = 0; s < kUStages; ++s) mbar_init(&bars[w][s], 1);
  }
  fence_mbar_init();
  __syncthreads();

  const int S_in = __ldg(p.seq_lens + b);
  const bool len_ok = S_in >= 1 && S_in <= max_slots;
  const int S = len_ok ? S_in : 0;  // an invalid length reads nothing: zero rows
  if (!len_ok && h == 0 && rank == 0 && tid == 0) report(p.status, WM_ERR_BOUNDS);
  const int nst = (S + STAGE_SLOTS - 1) / STAGE_SLOTS;
  const int npieces = C * NW, piece = rank * NW + warp;
  const int s0 = (int)((int64_t)piece * nst / npieces);
  const int nmine = (int)((int64_t)(piece + 1) * nst / npieces) - s0;

  T* myring = ring + warp * kUStages * RING_ELEMS;
  const uint64_t policy = l2_evict_first_policy();
  const T* kbase = reinterpret_cast<const T*>(p.k_pool) + (int64_t)h * p.P * HD;
  const T* vbase = reinterpret_cast<const T*>(p.v_pool) + (int64_t)h * p.P * HD;

  // Page-table window: lane i holds the page id of logical page win0 + i
  // (cur) and win0 + 32 + i (nxt); all lanes call page_of together.
  const int32_t* ptab = p.page_table + (int64_t)b * p.max_pages;
  int win0 = -64, pg_cur = -1, pg_nxt = -1;
  auto load_pg = [&](int lp) -> int { return lp < p.max_pages ? __ldg(ptab + lp) : -1; };
  auto page_of = [&](int lp, int lane_off) -> int {
    if (lp < win0 || lp >= win0 + 64) {
      win0 = lp;
      pg_cur = load_pg(lp + lane);
      pg_nxt = load_pg(lp + 32 + lane);
    } else if (lp >= win0 + 32) {
      win0 += 32;
      pg_cur = pg_nxt;
      pg_nxt = load_pg(win0 + 32 + lane);
    }
    const int idx = lp + lane_off - win0;  // 0 .. 63
    const int a = __shfl_sync(FULLMASK, pg_cur, idx & 31);
    const int c = __shfl_sync(FULLMASK, pg_nxt, idx & 31);
    return idx < 32 ? a : c;
  };

  // Copy stage s of the unit (the i-th of this warp) into ring slot i % S.
  auto issue = [&](int s) {
    const int buf = (s - s0) % kUStages;
    T* kd = myring + buf * RING_ELEMS;
    T* vd = kd + K_ELEMS;
    uint64_t* bar = &bars[warp][buf];
    const int s_begin = s * STAGE_SLOTS;
    attn_detail::copy_stage<MATH, T, HD, STAGE_SLOTS>(p, kbase, vbase, s_begin, S, kd, vd, bar,
                                                      &masks[warp][buf], 0u, policy, lane, page_of, []() {});
  };

  int issued = 0;
  for (; issued < nmine && issued < kUStages; ++issued) issue(s0 + issued);
  if (early) asm volatile("griddepcontrol.wait;" ::: "memory");

  // ---- stream this warp's stages
  constexpr int VRUN = CopyShape<MATH, STAGE_SLOTS>::kVRun;
  const int log2R = __ffs(min(p.P, VRUN)) - 1;  // mask bit of a slot = slot >> this
  const uint64_t all_pages = (1ull << (STAGE_SLOTS >> log2R)) - 1ull;
  MATH st;
  st.reset();
  // the unit's G query rows, read through L2 after the dependency wait (the
  // previous grid may have written them)
  if (nmine > 0)
    st.template load_q<true>(reinterpret_cast<const T*>(p.q) + ((int64_t)b * p.Hq + h * G) * HD, lane);
  bool alive = true;
  int done = 0;  // stages consumed
  for (; done < nmine && alive; ++done) {
    const int buf = done % kUStages;
    if (!__all_sync(FULLMASK, mbar_wait(&bars[warp][buf], (done / kUStages) & 1))) {
      if (lane == 0) report(p.status, WM_ERR_TIMEOUT);
      alive = false;
      break;
    }
    const int s = s0 + done;
    const int valid_slots = S - s * STAGE_SLOTS;
    const uint64_t mask = masks[warp][buf];
    const T* Ks = myring + buf * RING_ELEMS;
    const T* Vs = Ks + K_ELEMS;
    if (valid_slots >= STAGE_SLOTS && mask == all_pages)
      st.template consume<true>(Ks, Vs, lane, p.qscale, valid_slots, mask, log2R);
    else
      st.template consume<false>(Ks, Vs, lane, p.qscale, valid_slots, mask, log2R);
    __syncwarp();  // every lane is done with this ring slot
    if (issued < nmine) issue(s0 + issued++);
  }
  if (!alive) {
    // a copy never landed: wait (bounded) for what is still in flight and
    // contribute nothing
    if (lane == 0)
      for (int y = done; y < issued; ++y) mbar_wait(&bars[warp][y % kUStages], (y / kUStages) & 1);
    __syncwarp();
    st.reset();
  }

  // ---- merge the lanes of the warp, then store the warp's state in its
  // (idle) ring
  st.finish();
  st.store_state(reinterpret_cast<float*>(myring), lane);
  __syncthreads();

  // ---- merge the CTA's NW warp states, element by element
  T* outp = reinterpret_cast<T*>(p.out) + ((int64_t)b * p.Hq + h * G) * HD;
  auto warp_rec = [&](int w) -> const float* {
    return reinterpret_cast<const float*>(ring + w * kUStages * RING_ELEMS);
  };
  for (int e = tid; e < E; e += NW * 32) {
    const int g = e / HD;
    float mw[NW];
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      mw[w] = warp_rec(w)[E + 2 * g];
      M = fmaxf(M, mw[w]);
    }
    float Ls = 0.f, O = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float wt = mw[w] == -INFINITY ? 0.f : exp2f(mw[w] - M);
      Ls = fmaf(wt, warp_rec(w)[E + 2 * g + 1], Ls);
      O = fmaf(wt, warp_rec(w)[e], O);
    }
    if (C == 1) {
      outp[e] = Elem<T>::from_f(O * (Ls > 0.f ? 1.f / Ls : 0.f));
    } else {
      crec[e] = O;
      if (e == g * HD) {
        crec[E + 2 * g] = M;
        crec[E + 2 * g + 1] = Ls;
      }
    }
  }
  if (C == 1) return;

  // ---- merge the cluster's C CTA states: CTA `rank` finishes 1/C of the
  // unit's outputs, reading every CTA's state through distributed shared
  // memory; the second barrier keeps each CTA's shared memory alive until
  // every reader is done
  cluster.sync();
  const float* cr[kAttnUnitMaxCluster];
#pragma unroll
  for (int c = 0; c < kAttnUnitMaxCluster; ++c) cr[c] = c < C ? cluster.map_shared_rank(crec, c) : crec;
  const int e0 = rank * E / C, e1 = (rank + 1) * E / C;
  for (int e = e0 + tid; e < e1; e += NW * 32) {
    const int g = e / HD;
    float mq[kAttnUnitMaxCluster], lq[kAttnUnitMaxCluster], oq[kAttnUnitMaxCluster];
#pragma unroll
    for (int c = 0; c < kAttnUnitMaxCluster; ++c) {
      mq[c] = c < C ? cr[c][E + 2 * g] : -INFINITY;
      lq[c] = c < C ? cr[c][E + 2 * g + 1] : 0.f;
      oq[c] = c < C ? cr[c][e] : 0.f;
    }
    float M = -INFINITY;
#pragma unroll
    for (int c = 0; c < kAttnUnitMaxCluster; ++c) M = fmaxf(M, mq[c]);
    float Ls = 0.f, O = 0.f;
#pragma unroll
    for (int c = 0; c < kAttnUnitMaxCluster; ++c) {
      const float wt = mq[c] == -INFINITY ? 0.f : exp2f(mq[c] - M);
      Ls = fmaf(wt, lq[c], Ls);
      O = fmaf(wt, oq[c], O);
    }
    outp[e] = Elem<T>::from_f(O * (Ls > 0.f ? 1.f / Ls : 0.f));
  }
  cluster.sync();
}

template <typename T, int HD, int G, int SB, int NW, bool MMA = attn_uses_mma(kDtype<T>, HD, G)>
inline cudaError_t launch_unit_t(const AttnParams& p, int units, int cluster, size_t smem,
                                 cudaStream_t stream) {
  static size_t smem_set[kSmemOptDevices] = {};
  auto kern = decode_attn_unit_kernel<T, HD, G, SB, NW, MMA>;
  if (cudaError_t e = opt_in_smem(kern, smem, smem_set); e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)units * (unsigned)cluster);
  cfg.blockDim = dim3(NW * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

// Clusters of `cluster` CTAs that can be resident at once (0: unknown).
template <typename T, int HD, int G, int SB, int NW, bool MMA = attn_uses_mma(kDtype<T>, HD, G)>
inline int max_clusters_t(int cluster, size_t smem) {
  auto kern = decode_attn_unit_kernel<T, HD, G, SB, NW, MMA>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster * 64u);
  cfg.blockDim = dim3(NW * 32);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

template <typename T, int HD, int SB>
inline int max_clusters_g(int G, int warps, int cluster, size_t smem) {
  if (warps != 4 && warps != 8) return 0;
  switch (G) {
    case 1: return warps == 4 ? max_clusters_t<T, HD, 1, SB, 4>(cluster, smem) : 0;
    case 2:
      if (warps != 4) return 0;
      if constexpr (attn_unit_either(kDtype<T>, HD, 2)) {  // as many as fit either way
        const int a = max_clusters_t<T, HD, 2, SB, 4>(cluster, smem);
        const int b = max_clusters_t<T, HD, 2, SB, 4, true>(cluster, smem);
        return a < b ? a : b;
      }
      return max_clusters_t<T, HD, 2, SB, 4>(cluster, smem);
    case 4:
      if constexpr (sizeof(T) == 2)
        if (warps == 4) return max_clusters_t<T, HD, 4, SB, 4>(cluster, smem);
      return warps == 8 ? max_clusters_t<T, HD, 4, SB, 8>(cluster, smem) : 0;
    case 8:
      if constexpr (sizeof(T) == 2)
        if (warps == 4) return max_clusters_t<T, HD, 8, SB, 4>(cluster, smem);
      return warps == 8 ? max_clusters_t<T, HD, 8, SB, 8>(cluster, smem) : 0;
    default: return 0;
  }
}

template <typename T, int HD, int SB>
inline cudaError_t launch_unit_g(const AttnParams& p, int G, int warps, int units, int cluster, size_t smem,
                                 cudaStream_t s) {
  if (warps != 4 && warps != 8) return cudaErrorInvalidValue;
  switch (G) {
    case 1: return warps == 4 ? launch_unit_t<T, HD, 1, SB, 4>(p, units, cluster, smem, s) : cudaErrorInvalidValue;
    case 2:
      if constexpr (attn_unit_either(kDtype<T>, HD, 2))
        if (warps == 4 && attn_unit_mma(kDtype<T>, HD, 2, p.P, (int64_t)p.max_pages * p.P))
          return launch_unit_t<T, HD, 2, SB, 4, true>(p, units, cluster, smem, s);
      return warps == 4 ? launch_unit_t<T, HD, 2, SB, 4>(p, units, cluster, smem, s) : cudaErrorInvalidValue;
    case 4:
      if constexpr (sizeof(T) == 2)
        if (warps == 4) return launch_unit_t<T, HD, 4, SB, 4>(p, units, cluster, smem, s);
      return warps == 8 ? launch_unit_t<T, HD, 4, SB, 8>(p, units, cluster, smem, s) : cudaErrorInvalidValue;
    case 8:
      if constexpr (sizeof(T) == 2)
        if (warps == 4) return launch_unit_t<T, HD, 8, SB, 4>(p, units, cluster, smem, s);
      return warps == 8 ? launch_unit_t<T, HD, 8, SB, 8>(p, units, cluster, smem, s) : cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace attn_unit_detail

// Per-dtype dispatch of the unit split (one translation unit each); the
// max_clusters entry points return 0 for an unsupported shape or no device.
cudaError_t launch_attn_unit_bf16(const AttnParams& p, int stage_bytes, int d, int G, int warps, int units,
                                  int cluster, size_t smem, cudaStream_t s);
cudaError_t launch_attn_unit_f32(const AttnParams& p, int stage_bytes, int d, int G, int warps, int units,
                                 int cluster, size_t smem, cudaStream_t s);
int attn_unit_max_clusters_bf16(int stage_bytes, int d, int G, int warps, int cluster, size_t smem);
int attn_unit_max_clusters_f32(int stage_bytes, int d, int G, int warps, int cluster, size_t smem);

}  // namespace wm
