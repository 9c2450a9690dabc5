// Launch description of the tensor-core scoring path (score_tc_impl.cuh).
#pragma once

#include <cuda.h>
#include <cuda_fp16.h>

#include "ckv_internal.cuh"

namespace ckv {
namespace tc {

constexpr int kMaxTc = 16;          // trajectories per launch (tensor maps travel as parameters)
constexpr int kRowsPerTile = 128;   // probe rows per MMA tile
constexpr int kTileTokens = 128;    // tokens per MMA tile
constexpr int kSlot = 16;           // tokens per page slot
constexpr int kListSlotsPerItem = 64;  // slots per work item of the pruned page pass
constexpr int kSlotsPerItem = 128;  // 16-token slots per pass-B work item
constexpr int kPartsPerItem = 1;    // pass-A partials per work item (the two softmax groups merged)
constexpr int kPartialRing = 4;     // partial slots (items) per flash CTA of the fused launch
constexpr int kMaxFusedCtas = 256;  // bound on the fused launch's flash CTAs (workspace sizing)
constexpr int kFusedItemsPerSlice = 32;    // flash items per slice in the fused launch (chunking target)
constexpr double kFusedFlashShare = 0.55;  // share of the SMs that run the flash pass in the fused launch
constexpr int kCounterStride = 32;  // per-slice counters of the fused launch, one 128-byte line each

struct TcMaps {
  CUtensorMap q;             // Q as [M*Hq*W rows][d], box 64 x 128
  CUtensorMap k, v;          // K, V as [M][H][S][d], box 64 x 128 x 1 x 1
  CUtensorMap kb[3], vb[3];  // the same with 16-, 32- and 64-row boxes (runs of page slots)
};

// Per-trajectory facts computed once per call by the prep kernel.
struct TcPrep {
  int vis_all;  // leading resident tokens visible to every probe row
  int nitem;    // entries of the item table that hold pages
  int pad[2];
};

// A unit is one 128-row tile of probe rows of one (trajectory, selected
// layer, KV head) slice: unit (li * H + kvh) * nrt + rt of its trajectory.
// Workspace of the pruned page pass, per trajectory; null pointers when the
// launch is not pruned.
struct TcPrune {
  uint2 *cuts;         // [4 ntile]: per 32 tokens, {page starts and ends, page ends} as bit masks
  int2 *tile;          // [ntile]: {index of the tile's first piece, 1 if a page covers its last token}
  int32_t *piece_off;  // [P + 1]: first piece of every page (a page has one piece per tile it touches)
  __half *pieces;      // [units][npiece][128]: log2 of the row's exp-sum over the piece, rounded up
  __half *vnorm;       // [slices][128 ntile]: upper bound of every token's |v|
  float4 *aux;         // [units][128]: {final max (base 2), exp-sum, |o|, 0} of every probe row
  float *bound;        // [units][P]: upper bound of the page's effect on the unit's rows
  unsigned long long *seed;  // [P]: {bound bits, unit} of the unit with the largest bound (0: no effect)
  int32_t *list;       // [units][cap]: slots of the unit's pages that are to be scored
  int npiece, cap;
};

struct TcTraj {
  const int32_t *pos, *qpos, *ps, *pl;
  int32_t *slot_off;  // workspace [P + 1]
  int4 *items;        // workspace [nbitem][2]: {E0, E1, slot0, nslot}, {npages, 0, 0, 0}
  int4 *slot_tab;     // workspace [ceil(S/16) + P]: {tok0, nv, page, first | last << 1}
  TcPrep *prep;       // workspace
  int32_t *nvis_w;    // workspace [W]: resident tokens visible to each window position
  float *stats;       // [M][Hq][W][d + 4]
  float *R;           // [P]
  float *headR;       // [M][Hq][P] or null
  int S, W, P, nchunk, nrt, nbitem;
  TcPrune pr;
};

struct TcLaunch {
  TcMaps maps[kMaxTc];
  TcTraj t[kMaxTc];
  int n_traj, M, H, Hq, g, n_layers, chunk_len, slots_per_item;
  int from_stats;  // the stats are the caller's: no flash pass, no combine
  float scale_log2;
  float *partials;  // [items_a or n_a * kPartialRing][128][d + 4]: one partial per work item
  int item_off_a[kMaxTc + 1], item_off_b[kMaxTc + 1], row_off[kMaxTc + 1];
  // fused launch: CTAs [0, n_a) run the flash pass, the rest the page pass
  int fused;  // 1: one cooperative launch of both passes (set by the caller; needs !from_stats)
  int n_a;    // set by launch_score_tc
  int slice_off[kMaxTc + 1];  // (trajectory, selected layer, KV head) slices: prefix per trajectory
  uint32_t *a_done;           // workspace [slices][kCounterStride]: flash-pass warps done with their partials
  uint32_t *merged;           // workspace [slices][kCounterStride]: merge warps done with their rows
  // pruned page pass (set by the caller): only the pages of a unit whose
  // bound can raise R are scored
  int prune;
  int unit_off[kMaxTc + 1];   // units: prefix per trajectory
  int bound_off[kMaxTc + 1];  // blocks of bound_kernel: prefix per trajectory
  int seed_off[kMaxTc + 1];   // blocks of seed_kernel
  int4 *list_items;           // workspace: {unit, first entry of its list, entries, pages} of every work item
  uint8_t layer_ids[kMaxLayers];
};

// Bytes of workspace of the pruned page pass for one trajectory of up to S
// tokens and P pages (monotone in S, P, slices and nrt), and of the shared
// part (list_items) that it adds.
size_t prune_bytes(int S, int P, int slices, int nrt);
size_t prune_item_bytes(int S, int P, int slices, int nrt);
// Lays the region out at `base`.
void prune_layout(TcPrune &p, char *base, int S, int P, int slices, int nrt);
// The page pass is pruned when the pages average at least kMinPageTokens
// tokens (bounds the bookkeeping, which is per page and row: with 36 layers,
// 8 KV heads and 16K + 2K tokens the call takes 5.8 ms against 15.6 ms with
// the full pass for pages of 2 tokens, 1.48 against 2.24 ms for 32, 1.76
// against 1.99 ms for 256), and when the launch has kMinPruneWork (unit,
// token) pairs: below, the extra launches cost more than they save.  Pruned
// against full, us, 128 probe rows a unit: 2^18.1 pairs (1 layer of 16K + 2K
// tokens) 176 and 126, 2^19.1 (2 layers) 214 and 210, 2^19.6 (36 layers of
// 1.2K + 0.3K) 379 and 343, 2^20.1 (4 layers of 16K + 2K) 287 and 332, 2^20.4
// (64 layers of 1.2K + 0.3K) 608 and 579, 2^21.3 (36 layers of 4K + 0.5K) 684
// and 870.  32 of a unit's 128 rows: 2^18.1 201 and 149, 2^19.1 251 and 255,
// 2^19.6 300 and 336, 2^20.1 336 and 392, 2^20.4 458 and 560, 2^21.3 648 and 1,000.
// What is dropped depends on the data, which no rule here sees.  Where
// nothing is (keys all alike) the sums, bounds and lists come on top of the
// full pass: one cache of 18K tokens, 36 layers, in pages of 32 1,742 against
// 1,585 us, of 16 2,439 against 2,133, of 100 and 250 1,602 against 1,490, of
// 2 and 3 11.9 against 9.4 ms; 8 layers of 128K, 512 rows a KV head, 7.45
// against 6.9 ms.  With random keys 1,298, 1,196, 1,604 us, 3.3 and 6.8 ms.
constexpr int kMinPageTokens = 2;
constexpr int64_t kMinPruneWork = 1 << 20;

// The kernels for one head width.
namespace d128 {
bool build_maps(TcMaps &maps, const TrajDev &t, int M, int H, int Hq);
cudaError_t launch_score_tc(TcLaunch &L, WsHeader *hdr, cudaStream_t stream, int sm_count);
}  // namespace d128
namespace d64 {
bool build_maps(TcMaps &maps, const TrajDev &t, int M, int H, int Hq);
cudaError_t launch_score_tc(TcLaunch &L, WsHeader *hdr, cudaStream_t stream, int sm_count);
}  // namespace d64
inline bool build_maps(int d, TcMaps &maps, const TrajDev &t, int M, int H, int Hq) {
  return d == 64 ? d64::build_maps(maps, t, M, H, Hq) : d128::build_maps(maps, t, M, H, Hq);
}
inline cudaError_t launch_score_tc(int d, TcLaunch &L, WsHeader *hdr, cudaStream_t stream, int sm_count) {
  return d == 64 ? d64::launch_score_tc(L, hdr, stream, sm_count) : d128::launch_score_tc(L, hdr, stream, sm_count);
}
// Flash-pass CTAs of a fused launch on sm_count SMs (the rest run the page pass).
int fused_flash_ctas(const TcLaunch &L, int sm_count);
// Chunk length (tokens) of the fused launch for caches of up to max_tokens
// tokens and max_row_tiles 128-row tiles of probe rows per slice.
int fused_chunk_len(int max_tokens, int max_row_tiles);

}  // namespace tc
}  // namespace ckv
