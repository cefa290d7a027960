// Launch interfaces between the C-ABI layer (wm_api.cu) and the kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "wm.h"

namespace wm {

// Opt kernel `kern` into `smem` bytes of dynamic shared memory on the current
// device (the limit is a per-device attribute of the function).  `done`
// holds, per device, the largest value set so far.
constexpr int kSmemOptDevices = 64;
template <typename Kern>
inline cudaError_t opt_in_smem(Kern kern, size_t smem, size_t (&done)[kSmemOptDevices]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  const bool cached = dev >= 0 && dev < kSmemOptDevices;
  if (cached && smem <= done[dev]) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && cached) done[dev] = smem;
  return e;
}

// ------------------------------------------------------------ attention
struct AttnParams {
  const void* k_pool;     // channel c(layer) base of the K pool
  const void* v_pool;     // channel c(layer) base of the V pool
  const void* q;          // [B][Hq][d]
  void* out;              // [B][Hq][d]
  const int32_t* page_table;
  const int32_t* seq_lens;
  float* part;            // [2][max_chunks] records of attn_part_rec(G, d) floats: the
                          // partial of the first piece (side 0) / last piece (side 1) of
                          // each chunk that belongs to a unit crossing a chunk boundary
                          // ([G][d] unnormalised outputs, (max, sum) per query head in
                          // log2 units, then a published flag, zero between launches)
  int32_t* counters;      // [0]: chunk counter; [1 + g]: arrival tickets of the unit whose
                          // first piece ends chunk g; zero between launches
  int32_t* status;
  int64_t page_stride;    // elements between consecutive physical pages
  int32_t B, Hq, Hkv, P, log2P, num_pages, max_pages;
  int32_t chunk_stages;   // stages per work chunk (0: one chunk per warp)
  int32_t max_chunks;     // partial slots per side
  int32_t inputs_ready;   // the previous grid wrote no cache, table, length or workspace
  int32_t epoch;          // nonzero tag of this call: a record is published when its
                          // flag holds this value (a stale word from another call or
                          // layout never matches)
  float qscale;           // log2(e) / sqrt(d)
};

// Resident CTAs per SM the attention kernel is built for: 4 with 4 KB stages
// and one query head per kv head, else 2 (GQA keeps G query rows per lane).
// The planner uses 8 KB stages only.
constexpr int attn_ctas_per_sm(int stage_bytes, int G) { return stage_bytes == 4096 && G == 1 ? 4 : 2; }

// Floats per partial record: G*d outputs, (max, sum) per head, a "published"
// flag word, padded to 16 bytes so that consecutive records can be moved with
// one bulk copy.
constexpr int attn_part_rec(int G, int d) { return G * d + (2 * G + 1 + 3) / 4 * 4; }

// Launches whose stage math runs on the tensor cores (attn_mma.cuh): bf16
// with four or eight query heads per kv head, or two of 96 (69 launches in 0.92 of
// the time on the CUDA cores).  Two of 128 were faster on the CUDA cores, with the 8 warps
// per SM that its stages leave room for (step of 8 layers, 4 ragged sequences up to 4096,
// 16/8 heads: 115 us, 127 on the tensor cores).  Two of 64: see attn_unit_mma.  A stage of
// theirs is kAttnMmaPad bytes longer in shared memory.
constexpr bool attn_uses_mma(int dtype, int d, int G) {
  return dtype == WM_DT_BF16 && (G >= 4 || (G == 2 && d == 96));
}
constexpr int kAttnMmaPad = 64;

int attn_stage_slots(int stage_bytes, int dtype, int d);
int attn_warps_per_cta();
size_t attn_smem_bytes(int stage_bytes, int dtype, int d, int G, int B);
cudaError_t launch_decode_attn(const AttnParams& p, int stage_bytes, int dtype, int d, int G,
                               int grid, cudaStream_t s);
// Unit split (attn_unit.cuh): one cluster of `cluster` CTAs (<= 8) per
// (sequence, kv head) unit, `units` = B * Hkv clusters.
constexpr int kAttnUnitMaxCluster = 8;
int attn_unit_warps_per_cta(int stage_bytes, int G);  // 0: unsupported
// ... and of the unit split; its two query heads of 64 can run either way: V in two
// copies per stage (pages of more than 16 slots) costs what the tensor cores gain, so
// only where pages are that small or the units short.  (us, CUDA cores / tensor cores: six
// sequences of 162, 16 kv heads 5.4 / 5.0; three of up to 3687, 8, pages of 16: 8.9 / 8.6;
// nine of up to 4811, 4, pages of 64: 10.1 / 10.6; on stream-K 83 of up to 2776, 32: 218 /
// 229, and 34 of 617, 12: 18.4 / 19.3.)
constexpr bool attn_unit_either(int dtype, int d, int G) { return dtype == WM_DT_BF16 && d == 64 && G == 2; }
constexpr bool attn_unit_mma(int dtype, int d, int G, int page, int64_t max_slots) {
  return attn_uses_mma(dtype, d, G) || (attn_unit_either(dtype, d, G) && (page <= 16 || max_slots <= 2048));
}
size_t attn_unit_smem_bytes(int stage_bytes, int dtype, int d, int G, int warps);
int attn_unit_max_clusters(int stage_bytes, int dtype, int d, int G, int warps, int cluster);
cudaError_t launch_decode_attn_unit(const AttnParams& p, int stage_bytes, int dtype, int d, int G,
                                    int warps, int units, int cluster, cudaStream_t s);

// ------------------------------------------------------------ prefill attention
struct PrefillLaunch {
  const void* q;              // [B][Tq][Hq][d] bf16
  const int32_t* pos;         // [B][Tq] token position of each query row
  const int32_t* page_table;  // [B][max_pages]
  void* out;                  // [B][Tq][Hq][d] bf16
  int32_t* status;
  const void* k_pool;         // whole pools, all channels: [k][num_pages][Hkv][P][d]
  const void* v_pool;
  int32_t B, Tq, Hq, Hkv, d, k, chan, num_pages, max_pages, P;
};
cudaError_t launch_prefill_attn(const PrefillLaunch& L, int sms, cudaStream_t s);

// ------------------------------------------------------------ TMA tensor maps
// 2-D map of a row-major bf16 matrix [rows][cols] with a row pitch of
// pitch_elems elements (a multiple of 8), a box of 64 columns x box_rows
// rows and 128-byte swizzle; elements outside the matrix read as zero.
// `tm` points at a CUtensorMap.  False if the encoder is missing or refuses.
bool tma_available();
bool tma_map_bf16_2d(void* tm, const void* ptr, uint64_t rows, uint64_t cols, uint64_t pitch_elems,
                     uint32_t box_rows);

// ------------------------------------------------------------ KV pool (mix)
constexpr int kMaxRopeHalf = 64;  // d/2 for d <= 128

struct MixParams {
  // shape
  int32_t B, L, k, D, Hkv, d, p, Lp, P, log2P, num_pages, max_pages;
  float eps_rms, eps_qk;
  // inputs
  const void* h;                  // [B][L][D]
  const void* pre_g[2];
  const void* Wr[2];
  const void* br[2];
  const void* ch_g[2];
  const void* Wkv[2];
  const void* qk_g;
  const int32_t* page_table;
  const int32_t* slot;
  // cache
  void* k_pool;
  void* v_pool;
  // workspace
  float* inv_rms;                 // [B][L]
  void* xi;                       // [2][B][Lp*D] router inputs (dtype of the config)
  float* zpart;                   // [2][nsplit_r][B][k*L] router partial sums
  float* rope_cs;                 // [B][d/2][2] cos, sin at pos = slot - 1
  void* xop;                      // [2][k][B][D] normed channels, dtype
  float* proj;                    // [2][k][B][Hkv*d] projection outputs (fp32 path)
  float* ssq;                     // [2][k][mix_parts][B] sums of htilde^2 over parts of D (bf16)
  int32_t mix_parts;
  int32_t sms;
  int32_t nsplit_r;
  int32_t* status;
  double inv_freq[kMaxRopeHalf];  // theta^(-2i/d), computed on the host in fp64
};

struct MixWorkspace {
  size_t inv_rms, xi, zpart, rope_cs, xop, proj, total;
  int32_t nsplit_r;
};

MixWorkspace mix_workspace_layout(const wm_config& cfg, int32_t B, int sm_count);
cudaError_t launch_kv_mix(MixParams& p, int dtype, int sms, cudaStream_t s);
int kv_mix_launches(const MixParams& p, int dtype);  // kernels launch_kv_mix enqueues

// tcgen05 projection with the fused key/value epilogue, and the tcgen05
// router with split-K fp32 partials (bf16 only)
bool proj_tc_supported(const MixParams& p);
cudaError_t launch_proj_tc(const MixParams& p, cudaStream_t s);
int router_tc_splits(int k, int L, int Lp, int D, int sms);
cudaError_t launch_router_tc(const MixParams& p, cudaStream_t s);
// the same for groups of tokens (proj_rows.cu), from kRowsTokens tokens on
constexpr int kRowsTokens = 128;
bool proj_rows_supported(const MixParams& p);
cudaError_t launch_proj_rows(const MixParams& p, int sms, cudaStream_t s);
int router_rows_splits(int k, int L, int Lp, int D, int B, int sms);
cudaError_t launch_router_rows(const MixParams& p, int sms, cudaStream_t s);

}  // namespace wm
