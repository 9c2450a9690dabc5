// Tensor-core scoring for 128-channel heads (score_tc_impl.cuh), and what
// does not depend on the head width: workspace sizes of the pruned page pass
// and the shape of the fused launch.
#define CKV_TC_D 128
#define CKV_TC_NS d128
#include "score_tc_impl.cuh"

namespace ckv {
namespace tc {

namespace {
struct PruneSizes {
  size_t cuts, tile, piece_off, pieces, vnorm, aux, bound, seed, list;
  int npiece, cap;
};
PruneSizes prune_sizes(int S, int P, int slices, int nrt) {
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t ntile = ((size_t)S + kTileTokens - 1) / kTileTokens, units = (size_t)slices * nrt;
  const size_t p = (size_t)(P < S / kMinPageTokens ? P : S / kMinPageTokens);
  PruneSizes z;
  z.npiece = (int)(p + ntile);
  z.cap = (int)((size_t)S / kSlot + 1 + p);
  z.cuts = up(4 * ntile * sizeof(uint2));
  z.tile = up(ntile * sizeof(int2));
  z.piece_off = up((p + 1) * 4);
  z.pieces = up(units * z.npiece * kRowsPerTile * sizeof(__half));
  z.vnorm = up((size_t)slices * ntile * kTileTokens * sizeof(__half));
  z.aux = up(units * kRowsPerTile * sizeof(float4));
  z.bound = up(units * p * 4);
  z.seed = up(p * 8);
  z.list = up(units * z.cap * 4);
  return z;
}
}  // namespace

size_t prune_bytes(int S, int P, int slices, int nrt) {
  const PruneSizes z = prune_sizes(S, P, slices, nrt);
  return z.cuts + z.tile + z.piece_off + z.pieces + z.vnorm + z.aux + z.bound + z.seed + z.list;
}

size_t prune_item_bytes(int S, int P, int slices, int nrt) {
  const PruneSizes z = prune_sizes(S, P, slices, nrt);
  return (size_t)slices * nrt * ((size_t)z.cap / kListSlotsPerItem + 1) * sizeof(int4);
}

void prune_layout(TcPrune &p, char *base, int S, int P, int slices, int nrt) {
  const PruneSizes z = prune_sizes(S, P, slices, nrt);
  auto take = [&](size_t n) {
    char *at = base;
    base += n;
    return at;
  };
  p.cuts = reinterpret_cast<uint2 *>(take(z.cuts));
  p.tile = reinterpret_cast<int2 *>(take(z.tile));
  p.piece_off = reinterpret_cast<int32_t *>(take(z.piece_off));
  p.pieces = reinterpret_cast<__half *>(take(z.pieces));
  p.vnorm = reinterpret_cast<__half *>(take(z.vnorm));
  p.aux = reinterpret_cast<float4 *>(take(z.aux));
  p.bound = reinterpret_cast<float *>(take(z.bound));
  p.seed = reinterpret_cast<unsigned long long *>(take(z.seed));
  p.list = reinterpret_cast<int32_t *>(take(z.list));
  p.npiece = z.npiece;
  p.cap = z.cap;
}

int fused_chunk_len(int max_tokens, int max_row_tiles) {
  // about kFusedItemsPerSlice flash items per slice (row tiles included), at
  // least 512 tokens each, whole 128-token tiles
  const int64_t per = ((int64_t)max_tokens * max_row_tiles + kFusedItemsPerSlice - 1) / kFusedItemsPerSlice;
  const int64_t c = per < 512 ? 512 : per;
  return (int)((c + kTileTokens - 1) / kTileTokens * kTileTokens);
}

int fused_flash_ctas(const TcLaunch &L, int sm_count) {
  int na = (int)(sm_count * kFusedFlashShare + 0.5);
  if (const char *e = getenv("COMMITKV_FUSED_FLASH_CTAS")) na = atoi(e);  // tuning experiments
  const int items_a = L.item_off_a[L.n_traj], items_b = L.item_off_b[L.n_traj];
  if (items_b == 0) na = sm_count;
  na = na < 1 ? 1 : na > sm_count - 1 ? sm_count - 1 : na;
  // A partial slot is reused n_a * kPartialRing items later, after the slice of its
  // earlier item is merged.  That slice's items must all come earlier than
  // the reusing item (else the wait could depend on itself): n_a * kPartialRing
  // must cover the items of any slice.
  int nis_max = 1;
  for (int t = 0; t < L.n_traj; ++t) {
    const int nis = L.t[t].nchunk * L.t[t].nrt;
    nis_max = nis > nis_max ? nis : nis_max;
  }
  const int na_min = (nis_max + kPartialRing - 1) / kPartialRing;
  na = na < na_min ? na_min : na;
  return na < items_a ? na : items_a;
}

}  // namespace tc
}  // namespace ckv
