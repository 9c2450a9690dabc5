// Page deletion effects (Section 3.2, Eq. 6-8) on the 5th-generation tensor
// cores: bf16 K/V/Q, fp32 accumulation in tensor memory.  Compiled once per
// head width: CKV_TC_D = 128 (score_tc.cu) or 64 (score_tc64.cu).
//
//   pass A   persistent, warp-specialised flash forward over 128-token tiles
//            of a token chunk: S = Q K^T (tcgen05, TMEM), online softmax in
//            base 2 with a lazy max (O is rescaled only when the row max
//            grows by more than 2^8), O += P V; writes the
//            chunk's (max, sum, count, O) per probe row.
//   combine  merges a slice's chunk partials into the row stats
//            (m, l, n, o) of the whole cache.
//   prep     per trajectory, the prefix count of 16-token slots per page.
//   bounds   an upper bound of every page's effect on the 128 probe rows of
//            a unit, from the row sums over pages that pass A left (large
//            calls without maxima per head): pass B then scores only the
//            pages of a unit that can raise R, first those of the unit with
//            the largest bound, then those whose bound is above the effects
//            found.  On 36 layers of 16K + 2K tokens (pages of 32): page pass
//            1,495 us, instead bounds 57, lists 13, page pass over the rest
//            245, and pass A 900 -> 1,070 us for the sums; 32K + 4K: scoring
//            4.26 -> 2.55 ms.
//   pass B   persistent, over tiles of 8 slots: every page is loaded as
//            16-row TMA boxes into slots of its own, so one page's columns
//            never share a 16-wide MMA k-block with another page.
//            S = Q K_slots^T; e = exp(s - m) on the page's visible tokens;
//            U_E = sum_{i in E} e_i v_i by per-slot MMAs accumulating into
//            one of two 128-column TMEM accumulators; a separate epilogue
//            warpgroup reduces U_E to
//              r = ||U_E - S_E o|| / ((l - S_E) ||o||)      (Eq. 6 with a = e / l)
//            and max-reduces r over rows into R[E] (Eq. 7).
// Every mbarrier wait is bounded (1 s); on expiry the kernel records
// COMMITKV_ERR_TIMEOUT and all warps leave their loops.
#include <cudaTypedefs.h>
#include <stdlib.h>

#include "ckv_internal.cuh"
#include "sm103.cuh"
#include "score_tc.cuh"

namespace ckv {
namespace tc {
namespace CKV_TC_NS {
namespace {

using namespace ckv::sm103;

constexpr int D = CKV_TC_D;
constexpr int NH = D / 64;  // 64-channel halves of a tile (128-byte rows in shared memory)
constexpr int BM = 128;  // probe rows per tile (MMA M)
constexpr int BT = 128;  // KV rows per tile (MMA N of Q K^T, K of P V)
constexpr int NKB = D == 128 ? 3 : 5;  // K stages (pass B: with their slot tables)
constexpr int NVB = D == 128 ? 2 : 4;  // V stages
// P as bf16 terms: with 128 channels tensor memory has room for two (P to
// 2^-16, see split_pack32), with 64 for three (P to fp32's own precision,
// which the CUDA-core kernels for this width have as well).
constexpr int NP = D == 128 ? 2 : 3;
// The tensor cores' accumulation truncates: the output over hundreds of MMAs
// is off by 5e-6 to 1e-5.  With 64 channels the softmax threads have the
// registers to take every tile's P V out of tensor memory and add it up in
// fp32 (kRegO), and the row outputs are as exact as the CUDA-core kernels'.
constexpr bool kRegO = D == 64;
// Tensor memory: two S/P buffers of PW columns, then two accumulators of D.
// The softmax writes chunk c's P (32 tokens, 16 columns per term) at column
// 16 NP c and reads S from column S0 + 32 c: a chunk's P ends at or before
// the next chunk's S.
constexpr int PW = 64 * NP;
constexpr int S0 = PW - BT;
static_assert(2 * PW + 2 * D <= 512 && 3 * 16 * NP <= S0 + 3 * 32, "tensor memory layout");
constexpr int SLOT = 16;
constexpr int SLOTS = BT / SLOT;  // slots per pass-B tile
constexpr int NFIFO = 16;         // page-sum FIFO depth (>= 2 x SLOTS)
constexpr uint64_t kWait = 1000000000ull;
constexpr float kLazy = 8.0f;     // rescale O when the max grows by > 2^8
constexpr int kRing = kPartialRing;  // partial slots per flash CTA of the fused launch

constexpr uint32_t kHalf = BT * 128;  // one 64-channel half of a tile: 16 KB
constexpr uint32_t kTileBytes = NH * kHalf;

// ----------------------------------------------------------------- helpers
__device__ __forceinline__ int traj_of(const int32_t *off, int n, int item) {
  int t = 0;
  while (t + 1 < n && item >= off[t + 1]) ++t;
  return t;
}

__device__ __forceinline__ void tma4(void *dst, const CUtensorMap *m, int x, int tok, int h, int l,
                                     uint64_t *bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(x), "r"(tok), "r"(h), "r"(l), "r"(smem_addr(bar)), "l"(pol)
      : "memory");
}


// The boxes of all halves of a tile.
__device__ __forceinline__ void tma4_all(uint8_t *dst, const CUtensorMap *m, int tok, int h, int l, uint64_t *bar,
                                         uint64_t pol) {
#pragma unroll
  for (int x = 0; x < NH; ++x) tma4(dst + x * kHalf, m, 64 * x, tok, h, l, bar, pol);
}
__device__ __forceinline__ void tma_q(uint8_t *dst, const CUtensorMap *m, int row, uint64_t *bar, uint64_t pol) {
#pragma unroll
  for (int x = 0; x < NH; ++x) tma_load_2d(dst + x * kHalf, m, 64 * x, row, bar, pol);
}

// K-major operand tile (rows x D elements, 64-element halves): the
// descriptor of the 16-element k-step `ks`.
__device__ __forceinline__ uint64_t desc_kmajor(const uint8_t *tile, int ks) {
  return smem_desc(smem_addr(tile) + (ks >> 2) * kHalf + (ks & 3) * 32, 16, 1024, kSwizzle128B);
}
// MN-major B operand (V rows = k, D channels = n): k-step of 16 rows.
__device__ __forceinline__ uint64_t desc_v(const uint8_t *tile, int ks) {
  return smem_desc(smem_addr(tile) + ks * 2048, kHalf, 1024, kSwizzle128B);
}

// ============================================================== fused-launch plumbing
// Partial slot of a flash-pass item.  The two-launch path keeps one slot per
// item.  The fused launch keeps n_a * kRing slots: item i runs on CTA
// i mod n_a and takes slot i mod (n_a * kRing), last used by the same CTA's
// item i - n_a * kRing.
template <bool FUSED>
__device__ __forceinline__ float *part_ptr(const TcLaunch &L, int item, int h, int row) {
  const int64_t slot = FUSED ? (int64_t)(item % (L.n_a * kRing)) : (int64_t)item;
  return L.partials + ((slot * kPartsPerItem + h) * BM + row) * (D + 4);
}

// Index of an item's (trajectory, layer, KV head) slice in the per-slice counters.
template <class Item>
__device__ __forceinline__ int slice_of(const TcLaunch &L, const Item &it) {
  return (L.slice_off[it.t] + it.li * L.H + it.kvh) * kCounterStride;
}
__device__ __forceinline__ int items_per_slice(const TcLaunch &L, int t) { return L.t[t].nchunk * L.t[t].nrt; }

// Called by all 32 lanes of a warp: waits until *p >= target (an acquire
// load by every lane, so each lane's later reads see the writes released
// with the counter).  Bounded: gives up on the CTA's or the launch's abort
// flag, or after kWait, recording a timeout and raising both flags.
__device__ __forceinline__ bool warp_poll_geq(const uint32_t *p, uint32_t target, volatile int *abort_flag,
                                              WsHeader *hdr) {
  uint64_t t0 = 0;
  for (;;) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (__all_sync(0xffffffffu, v >= target)) return true;
    const bool stop = *abort_flag || *reinterpret_cast<volatile int32_t *>(&hdr->abort);
    const uint64_t now = now_ns();
    if (t0 == 0) t0 = now;
    const bool late = now - t0 > kWait;
    if (__any_sync(0xffffffffu, stop || late)) {
      if (late && (threadIdx.x & 31) == 0) {
        *abort_flag = 1;
        atomicExch(&hdr->abort, 1);
        record_error(hdr, COMMITKV_ERR_TIMEOUT, 12);
      }
      return false;
    }
    __nanosleep(512);
  }
}

// Partials of the fused launch are written once and read once soon after:
// kept in L2 over the streaming K and V, dropped first after their read.
__device__ __forceinline__ void st_keep(float *p, float4 v) {
  asm volatile(
      "{\n\t.reg .b64 pol;\n\tcreatepolicy.fractional.L2::evict_last.b64 pol, 1.0;\n\t"
      "st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, pol;\n\t}" ::"l"(p),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
      : "memory");
}
__device__ __forceinline__ float4 ld_once(const float *p) {
  float4 v;
  asm volatile(
      "{\n\t.reg .b64 pol;\n\tcreatepolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
      "ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], pol;\n\t}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p)
      : "memory");
  return v;
}

// Called by all 32 lanes after each wrote its part of a result: one
// release increment of *p for the warp.
__device__ __forceinline__ void signal_add(uint32_t *p, int lane) {
  __threadfence();
  __syncwarp();
  if (lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

template <bool FUSED>
__device__ __forceinline__ void merge_row(const TcLaunch &L, int t, int li, int kvh, int row, int lane);

// Upper bound of |v| of row `tok` of a V tile in shared memory.
__device__ __forceinline__ __half norm_bound(const uint8_t *tile, int tok) {
  __nv_bfloat162 acc[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) acc[k] = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll
  for (int c = 0; c < D / 8; ++c) {
    const uint4 w = *reinterpret_cast<const uint4 *>(tile + (c >> 3) * kHalf + sw128_offset(tok, c & 7));
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __nv_bfloat162 v2 = *reinterpret_cast<const __nv_bfloat162 *>(&x[k]);
      acc[k] = __hfma2(v2, v2, acc[k]);
    }
  }
  float n2 = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) n2 += __low2float(acc[k]) + __high2float(acc[k]);
  return __float2half_ru(sqrtf(n2 * 1.07f) + 2e-18f);
}

// ============================================================== pass A
// Two softmax warpgroups take alternate tiles of a chunk (global tile g goes
// to warpgroup g & 1), each with its own S/P buffer, running max, sum and
// output accumulator, so one warpgroup's softmax overlaps the other's MMAs.
// TMEM columns: S/P buffer b at PW b (after the softmax reads a 32-column
// chunk of S it overwrites columns already read with 16 columns of each of
// P's terms), O_b at 2 PW + D b.  At the end of an item the two warpgroups
// merge their states in the CTA and write one partial.
struct SmemA {
  alignas(1024) uint8_t q[kTileBytes];
  alignas(1024) uint8_t k[NKB][kTileBytes];
  alignas(1024) uint8_t v[NVB][kTileBytes];
  int pos[2][4][BT];  // per softmax warp: positions of the current tile
  float4 gs[2][4][BM];  // SUMS: per S/P buffer, 32-column chunk and row, the sums of the chunk's groups of eight columns
  float mused[2][BM];   // SUMS: per S/P buffer and row, the reference max of P
  float4 pub[BM];     // fused launch: warpgroup 1's (reference max, sum, count, true max) of the item, per row
  uint64_t q_full, q_empty, k_full[NKB], k_empty[NKB], v_full[NVB], v_empty[NVB], s_full[2], s_empty[2], p_full[2],
      o_full[2], o_empty[2], drain, drain2, pub_full, pub_empty;
  uint32_t tmem;
  int abort_flag;
};

struct ItemA {
  int t, l, kvh, rt, c, li;
};

__device__ __forceinline__ ItemA decode_a(const TcLaunch &L, int item) {
  ItemA it;
  it.t = traj_of(L.item_off_a, L.n_traj, item);
  const TcTraj &tr = L.t[it.t];
  int local = item - L.item_off_a[it.t];
  it.rt = local % tr.nrt;
  local /= tr.nrt;
  it.c = local % tr.nchunk;
  local /= tr.nchunk;
  it.kvh = local % L.H;
  it.li = local / L.H;
  it.l = L.layer_ids[it.li];
  return it;
}

// TMEM column of the 8 packed P columns of term `term` (hi first) of k-step ks inside S/P buffer b.
__device__ __forceinline__ uint32_t p_col(int b, int ks, int term) {
  return b * PW + 16 * NP * (ks >> 1) + 8 * (ks & 1) + 16 * term;
}

// Issues S[b] = Q K^T for one tile (a k-step per 16 channels).
__device__ __forceinline__ void issue_qk(uint32_t tm, const uint8_t *q, const uint8_t *k, int b) {
  const uint32_t idesc = idesc_bf16_f32(BM, BT, 0, 0);
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks)
    mma_bf16(tm + b * PW + S0, desc_kmajor(q, ks), desc_kmajor(k, ks), idesc, ks > 0);
}

// Issues D (+)= P[:, 16 ks .. 16 ks + 15] V[16 ks .. 16 ks + 15, :] with P as
// its NP terms in TMEM buffer b; `first` overwrites D.
__device__ __forceinline__ void issue_pv_step(uint32_t tm, uint32_t d_col, const uint8_t *v, int b, int ks,
                                              bool first) {
  const uint32_t idesc = idesc_bf16_f32(BM, D, 0, 1);
  uint64_t bd = desc_v(v, ks);
#pragma unroll
  for (int t = 0; t < NP; ++t) mma_bf16_ts(tm + d_col, tm + p_col(b, ks, t), bd, idesc, (first && t == 0) ? 0u : 1u);
}

// Stores the terms of 32 tokens' P (chunk c of the buffer at `buf`).
__device__ __forceinline__ void store_p(uint32_t buf, int c, float (&x)[32]) {
  if constexpr (NP == 2) {
    uint32_t pk[32];
    split_pack32(x, pk);
    tmem_st32(buf + 32 * c, pk);
  } else {
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      uint32_t pk[16];
      split_term32(x, pk, t + 1 == NP);
      tmem_st16(buf + 16 * NP * c + 16 * t, pk);
    }
  }
}

// Two exponentials 2^(x scale + bias), the arguments in one instruction.
__device__ __forceinline__ void exp2_pair(float *x, float2 scale, float2 bias) {
  const float2 t = ffma2(make_float2(x[0], x[1]), scale, bias);
  x[0] = fast_exp2(t.x);
  x[1] = fast_exp2(t.y);
}
// Sum of eight values in packed pairs.
__device__ __forceinline__ float sum8(const float *x) {
  const float2 a = fadd2(make_float2(x[0], x[1]), make_float2(x[2], x[3]));
  const float2 b = fadd2(make_float2(x[4], x[5]), make_float2(x[6], x[7]));
  const float2 c = fadd2(a, b);
  return c.x + c.y;
}

// log2 on the special-function unit (log2 0 = -inf).
__device__ __forceinline__ float fast_log2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// SUMS: also what the pruned page pass needs: log2 of every row's exp-sum
// over every page (one piece per tile that the page touches) and an upper
// bound of every token's |v|.
template <bool FUSED, bool SUMS>
__device__ __forceinline__ void flash_body(const TcLaunch &L, WsHeader *hdr, uint8_t *smem_raw, const int cta,
                                           const int ncta) {
  SmemA &sm = *reinterpret_cast<SmemA *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int n_items = L.item_off_a[L.n_traj];
  volatile int *abort_flag = &sm.abort_flag;

  if (threadIdx.x == 0) {
    sm.abort_flag = 0;
    mbar_init(&sm.q_full, 1);
    mbar_init(&sm.q_empty, 1);
    for (int s = 0; s < NKB; ++s) {
      mbar_init(&sm.k_full[s], 1);
      mbar_init(&sm.k_empty[s], 1);
    }
    for (int s = 0; s < NVB; ++s) {
      mbar_init(&sm.v_full[s], 1);
      mbar_init(&sm.v_empty[s], SUMS ? 5 : 1);  // P V and, with SUMS, the four warps of the page sums
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.s_full[b], 1);
      mbar_init(&sm.s_empty[b], SUMS ? 5 : 1);
      mbar_init(&sm.p_full[b], 4);
      mbar_init(&sm.o_full[b], 1);
      mbar_init(&sm.o_empty[b], 4);
    }
    mbar_init(&sm.drain, 1);
    mbar_init(&sm.drain2, 1);
    mbar_init(&sm.pub_full, 4);   // warpgroup 1's warps: the item's state is published
    mbar_init(&sm.pub_empty, 4);  // warpgroup 0's warps: the publication is consumed
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sm.tmem;

  // warpgroup 0: TMA producer, P V issuer, Q K^T issuer, one idle warp; 1 and
  // 2: softmax of the even and the odd tiles; 3 (SUMS): page sums and token norms.  Register
  // budget per thread: 104 + 2 x 200 = the launch's 3 x 168, with SUMS
  // 72 + 2 x 176 + 88 = 4 x 128.
  if (warp < 4) {
    if (FUSED) regs_dec<48>();
    else if (SUMS) regs_dec<72>();
    else regs_dec<104>();
    if (warp == 0) {
      // ------------------------------------------------------------ TMA producer
      if (lane == 0) {
        uint64_t pol = policy_evict_normal();
        uint32_t it = 0, n_local = 0, n_k = 0, n_v = 0;  // tiles; Q, K and V copies issued
        bool stop = false;
        for (int item = cta; item < n_items && !stop; item += ncta, ++n_local) {
          if (*abort_flag) break;
          ItemA a = decode_a(L, item);
          const TcTraj &tr = L.t[a.t];
          const TcMaps &mp = L.maps[a.t];
          if (n_local > 0 && !mbar_wait(&sm.q_empty, (n_local - 1) & 1, kWait, abort_flag)) break;
          mbar_expect_tx(&sm.q_full, kTileBytes);
          int qrow = (a.l * L.Hq + a.kvh * L.g) * tr.W + a.rt * BM;
          tma_q(sm.q, &mp.q, qrow, &sm.q_full, pol);
          int t0 = a.c * L.chunk_len, t1 = min(tr.S, t0 + L.chunk_len);
          int ntile = (t1 - t0 + BT - 1) / BT;
          // K of tile g once Q K^T of tile g - NKB is done; V once P V of tile g - NVB is
          auto load_k = [&](uint32_t g, int tok) -> bool {
            int s3 = g % NKB;
            if (g >= NKB && !mbar_wait(&sm.k_empty[s3], ((g / NKB) - 1) & 1, kWait, abort_flag)) return false;
            mbar_expect_tx(&sm.k_full[s3], kTileBytes);
            tma4_all(sm.k[s3], &mp.k, tok, a.kvh, a.l, &sm.k_full[s3], pol);
            ++n_k;
            return true;
          };
          auto load_v = [&](uint32_t g, int tok) -> bool {
            int s2 = g % NVB;
            if (g >= NVB && !mbar_wait(&sm.v_empty[s2], ((g / NVB) - 1) & 1, kWait, abort_flag)) return false;
            mbar_expect_tx(&sm.v_full[s2], kTileBytes);
            tma4_all(sm.v[s2], &mp.v, tok, a.kvh, a.l, &sm.v_full[s2], pol);
            ++n_v;
            return true;
          };
          // K runs one tile ahead of V
          if (ntile > 0) stop = !load_k(it, t0);
          for (int j = 0; j < ntile && !stop; ++j) {
            if (j + 1 < ntile && !load_k(it + j + 1, t0 + (j + 1) * BT)) stop = true;
            else if (!load_v(it + j, t0 + j * BT)) stop = true;
          }
          it += ntile;
        }
        if (*abort_flag) {
          // let the copies already issued land before the CTA leaves
          for (uint32_t u = (n_k > NKB ? n_k - NKB : 0); u < n_k; ++u)
            mbar_wait_drain(&sm.k_full[u % NKB], (u / NKB) & 1, kWait);
          for (uint32_t u = (n_v > NVB ? n_v - NVB : 0); u < n_v; ++u)
            mbar_wait_drain(&sm.v_full[u % NVB], (u / NVB) & 1, kWait);
          if (n_local > 0) mbar_wait_drain(&sm.q_full, (n_local - 1) & 1, kWait);
        }
      }
  } else if (warp == 1) {
    // ------------------------------------------------------------ P V issuer
    if (lane == 0) {
      uint32_t it = 0;
      int uses0 = 0, uses1 = 0;  // items in which O_0 / O_1 have been filled so far
      bool ok = true;
      for (int item = cta; item < n_items && ok; item += ncta) {
        ItemA a = decode_a(L, item);
        const TcTraj &tr = L.t[a.t];
        int t0 = a.c * L.chunk_len, t1 = min(tr.S, t0 + L.chunk_len);
        int ntile = (t1 - t0 + BT - 1) / BT;
        for (int j = 0; j < ntile && ok; ++j) {
          uint32_t g = it + j;
          int s2 = g % NVB, b = g & 1;
          const bool first = j < 2, last = j + 2 >= ntile;  // of warpgroup b in this item
          // O_b of the previous item must have been read out before P V overwrites it
          const int ub = b ? uses1 : uses0;
          if (first && ub > 0 && !mbar_wait(&sm.o_empty[b], (ub - 1) & 1, kWait, abort_flag)) {
            ok = false;
            break;
          }
          if (!mbar_wait(&sm.p_full[b], (g >> 1) & 1, kWait, abort_flag) ||
              !mbar_wait(&sm.v_full[s2], (g / NVB) & 1, kWait, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < BT / 16; ++ks) issue_pv_step(tm, 2 * PW + b * D, sm.v[s2], b, ks, (first || kRegO) && ks == 0);
          mma_commit(&sm.s_empty[b]);
          mma_commit(&sm.v_empty[s2]);
          if (last) {
            mma_commit(&sm.o_full[b]);
            if (b) ++uses1;
            else ++uses0;
          }
        }
        it += ntile;
      }
      if (*abort_flag) {
        mma_commit(&sm.drain);  // every MMA issued by this thread has completed
        mbar_wait_drain(&sm.drain, 0, kWait);
      }
    }
    } else if (warp == 2) {
      // ------------------------------------------------------------ Q K^T issuer
      if (lane == 0) {
        uint32_t it = 0, n_local = 0;
        bool ok = true;
        for (int item = cta; item < n_items && ok; item += ncta, ++n_local) {
          ItemA a = decode_a(L, item);
          const TcTraj &tr = L.t[a.t];
          int t0 = a.c * L.chunk_len, t1 = min(tr.S, t0 + L.chunk_len);
          int ntile = (t1 - t0 + BT - 1) / BT;
          if (!mbar_wait(&sm.q_full, n_local & 1, kWait, abort_flag)) break;
          tc_fence_after();
          for (int j = 0; j < ntile && ok; ++j) {
            uint32_t g = it + j;
            int s3 = g % NKB, b = g & 1;
            if (!mbar_wait(&sm.k_full[s3], (g / NKB) & 1, kWait, abort_flag) ||
                (g >= 2 && !mbar_wait(&sm.s_empty[b], ((g >> 1) - 1) & 1, kWait, abort_flag))) {
              ok = false;
              break;
            }
            tc_fence_after();
            issue_qk(tm, sm.q, sm.k[s3], b);
            mma_commit(&sm.s_full[b]);
            mma_commit(&sm.k_empty[s3]);
            if (j + 1 == ntile) mma_commit(&sm.q_empty);  // every Q K^T of this item is issued
          }
          it += ntile;
        }
        if (*abort_flag) {
          mma_commit(&sm.drain2);  // every MMA issued by this thread has completed
          mbar_wait_drain(&sm.drain2, 0, kWait);
        }
      }
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------ softmax (warps 4..11)
    if (FUSED) regs_inc<208>();
    else if (SUMS) regs_inc<176>();
    else regs_inc<200>();
    const int hb = (warp - 4) >> 2;   // this warpgroup's tiles: g & 1 == hb
    const int wq = warp & 3;          // TMEM lane quarter of this warp
    const int row = wq * 32 + lane;   // probe row within the tile
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    const uint32_t o_col = 2 * PW + hb * D;
    int *posw = sm.pos[hb][wq];
    uint32_t it = 0;
    int uses = 0;  // items in which this warpgroup filled O_hb
    uint32_t n_it = 0;  // items of this CTA seen so far (fused launch)
    bool ok = true;
    for (int item = cta; item < n_items && ok; item += ncta) {
      ItemA a = decode_a(L, item);
      const TcTraj &tr = L.t[a.t];
      int rows = L.g * tr.W;
      int grow = a.rt * BM + row;  // row within the (layer, KV head) slice
      bool valid_row = grow < rows;
      const bool warp_rows = grow - lane < rows;  // the warp has a row of the slice
      int qp = valid_row ? tr.qpos[grow % tr.W] : -0x7fffffff;
      const int vis_all = tr.prep->vis_all;
      int t0 = a.c * L.chunk_len, t1 = min(tr.S, t0 + L.chunk_len);
      int ntile = (t1 - t0 + BT - 1) / BT;
      const int j0 = (hb - (int)it) & 1;  // first tile of this warpgroup in the item
      float *dst = part_ptr<FUSED>(L, item, hb, row);
      float m_used = -INFINITY, m_true = -INFINITY, lsum = 0.0f;
      float acc[kRegO ? D : 1];  // kRegO: the output, relative to m_used
#pragma unroll
      for (int i = 0; i < (kRegO ? D : 1); ++i) acc[i] = 0.0f;
      // adds the latest tile's P V (kRegO)
      auto take_o = [&]() {
#pragma unroll
        for (int c0 = 0; c0 < D; c0 += 32) {
          float y[32];
          tmem_ld32f(tm + lane_base + o_col + c0, y);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[(kRegO ? c0 + i : 0)] += y[i];
        }
      };
      int nvis = 0;
      for (int j = j0; j < ntile && ok; j += 2) {
        uint32_t g = it + j;
        const int b = hb;
        int tok0 = t0 + j * BT, nt = min(BT, t1 - tok0);
        // tiles inside the prefix every probe row sees need no position test
        const bool full = tok0 + nt <= vis_all;
        if (!full) {  // each warp keeps its own copy: no cross-warp barrier
          __syncwarp();
#pragma unroll
          for (int i = lane; i < BT; i += 32) posw[i] = i < nt ? tr.pos[tok0 + i] : 0x7fffffff;
          __syncwarp();
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[b], (g >> 1) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        // A warp without a probe row of the slice leaves its rows as they are:
        // rows are independent, and none of theirs is read.  (32 probe rows
        // of 128, contexts of 2K tokens: flash pass 470 -> 232 us.)
        if (!warp_rows) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.p_full[b]);
          continue;
        }
        // visibility of column i: inside the tile and, outside the prefix every
        // probe row sees, at or before the row's query position
        const bool simple = full && nt == BT;
        // row max over the tile, 32 columns at a time (the first sweep; the
        // second computes P)
        float mx[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mx[k] = -INFINITY;
        int cnt = simple ? BT : 0;
#pragma unroll 1
        for (int c0 = 0; c0 < BT; c0 += 32) {
          float x[32];
          tmem_ld32f(tm + lane_base + b * PW + S0 + c0, x);
          tmem_wait_ld();
          if (!simple) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              bool vis = c0 + i < nt && (full || posw[c0 + i] <= qp);
              x[i] = vis ? x[i] : -INFINITY;
              cnt += vis;
            }
          }
#pragma unroll
          for (int i = 0; i < 32; i += 8)
#pragma unroll
            for (int k = 0; k < 4; ++k) mx[k] = fmax3(mx[k], x[i + 2 * k], x[i + 2 * k + 1]);
        }
        float smax = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]);
        float mt = smax == -INFINITY ? smax : smax * L.scale_log2;
        nvis += cnt;
        m_true = fmaxf(m_true, mt);
        float m_new = fmaxf(m_used, mt);
        bool rescale = m_new > m_used + kLazy;  // false while both are -inf
        float alpha = (rescale && m_used != -INFINITY) ? exp2f(m_used - m_new) : 0.0f;
        if (rescale) m_used = m_new;
        if (j > j0) {
          // S of this tile is there, so the P V of this warpgroup's previous
          // tile is done (Q K^T waited for the buffer): O_hb is stable
          if constexpr (kRegO) {
            take_o();
            if (rescale) {
#pragma unroll
              for (int i = 0; i < D; ++i) acc[i] *= alpha;
            }
          } else if (__any_sync(0xffffffffu, rescale)) {
            float f = rescale ? alpha : 1.0f;
            // unrolled, every load of the row is in flight before the first
            // store waits (8 layers of 128K tokens, 512 rows a KV head:
            // 2,515 us rolled, 2,335 so); with SUMS the registers are short
            // (16K + 2K tokens in pages of 16: 842 rolled, 852 unrolled)
#pragma unroll(SUMS ? 1 : D / 32)
            for (int c0 = 0; c0 < D; c0 += 32) {
              uint32_t r[32];
              tmem_ld32(tm + lane_base + o_col + c0, r);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f);
              tmem_st32(tm + lane_base + o_col + c0, r);
            }
            tmem_wait_st();
          }
        }
        if (rescale) lsum *= alpha;
        const float neg_m = m_used == -INFINITY ? 0.0f : -m_used;
        const float2 scale2 = make_float2(L.scale_log2, L.scale_log2), neg_m2 = make_float2(neg_m, neg_m);
        // sweep 2: p = 2^(s c - m) on the visible columns (2^-inf = 0), the row
        // sum, and P's terms over S columns already read
        float ps = 0.0f;
#pragma unroll 1
        for (int c0 = 0; c0 < BT; c0 += 32) {
          float x[32];
          tmem_ld32f(tm + lane_base + b * PW + S0 + c0, x);
          tmem_wait_ld();
          if (!simple) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              bool vis = c0 + i < nt && (full || posw[c0 + i] <= qp);
              x[i] = vis ? x[i] : -INFINITY;
            }
          }
#pragma unroll
          for (int i = 0; i < 32; i += 2) exp2_pair(&x[i], scale2, neg_m2);
          float gs[4];  // sums of the four groups of eight columns
#pragma unroll
          for (int q = 0; q < 4; ++q) gs[q] = sum8(&x[8 * q]);
          ps += (gs[0] + gs[1]) + (gs[2] + gs[3]);
          if constexpr (SUMS) sm.gs[b][c0 / 32][row] = make_float4(gs[0], gs[1], gs[2], gs[3]);
          store_p(tm + lane_base + b * PW, c0 / 32, x);
        }
        if constexpr (SUMS) sm.mused[b][row] = m_used;
        tmem_wait_st();
        lsum += ps;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.p_full[b]);
      }
      if (!ok) break;
      {
        // One partial per item: warpgroup 1 publishes its (reference max,
        // sum, count, true max) and leaves its O in tensor memory; warpgroup
        // 0 rescales both outputs to the larger reference max, writes the
        // partial and hands both O accumulators back to the P V issuer.
        const bool mine = j0 < ntile;  // this warpgroup filled its O in this item
        if (hb == 1) {
          if (n_it > 0 && !__all_sync(0xffffffffu, mbar_wait(&sm.pub_empty, (n_it - 1) & 1, kWait, abort_flag))) {
            ok = false;
            break;
          }
          if (mine && !__all_sync(0xffffffffu, mbar_wait(&sm.o_full[1], uses & 1, kWait, abort_flag))) {
            ok = false;
            break;
          }
          if constexpr (kRegO) {
            if (mine) {  // the whole output back into tensor memory for warpgroup 0
              tc_fence_after();
              take_o();
#pragma unroll
              for (int c0 = 0; c0 < D; c0 += 32) {
                uint32_t y[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) y[i] = __float_as_uint(acc[c0 + i]);
                tmem_st32(tm + lane_base + o_col + c0, y);
              }
              tmem_wait_st();
            }
          }
          sm.pub[row] = make_float4(mine ? m_used : -INFINITY, lsum, (float)nvis, m_true);
          if (mine) ++uses;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.pub_full);
        } else {
          if (FUSED && item >= L.n_a * kRing) {
            // the partial slot was last used by this CTA's item kRing items
            // back: its slice must be merged before the slot is overwritten
            const ItemA pa = decode_a(L, item - L.n_a * kRing);
            if (!warp_poll_geq(&L.merged[slice_of(L, pa)], 4u * items_per_slice(L, pa.t), abort_flag, hdr)) {
              ok = false;
              break;
            }
          }
          if ((mine && !__all_sync(0xffffffffu, mbar_wait(&sm.o_full[0], uses & 1, kWait, abort_flag))) ||
              !__all_sync(0xffffffffu, mbar_wait(&sm.pub_full, n_it & 1, kWait, abort_flag))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const float4 o1 = sm.pub[row];
          const bool mine1 = (int)((1u - it) & 1u) < ntile;  // warpgroup 1 filled its O in this item
          const bool theirs = mine1 && o1.x != -INFINITY;
          const float m0 = mine ? m_used : -INFINITY;
          const float mr = fmaxf(m0, theirs ? o1.x : -INFINITY);
          const float f0 = m0 == -INFINITY ? 0.0f : exp2f(m0 - mr);
          const float f1 = theirs ? exp2f(o1.x - mr) : 0.0f;
          if constexpr (kRegO) {
            if (mine) take_o();
          }
#pragma unroll(kRegO ? D / 32 : 1)
          for (int c0 = 0; c0 < D; c0 += 32) {
            float x0[32], x1[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              x0[i] = kRegO ? acc[kRegO ? c0 + i : 0] : 0.0f;
              x1[i] = 0.0f;
            }
            if (mine && !kRegO) tmem_ld32f(tm + lane_base + 2 * PW + c0, x0);
            if (mine1) tmem_ld32f(tm + lane_base + 2 * PW + D + c0, x1);
            tmem_wait_ld();
            if (valid_row) {
#pragma unroll
              for (int i = 0; i < 32; i += 4) {
                const float4 v = make_float4(fmaf(x0[i], f0, theirs ? x1[i] * f1 : 0.0f),
                                             fmaf(x0[i + 1], f0, theirs ? x1[i + 1] * f1 : 0.0f),
                                             fmaf(x0[i + 2], f0, theirs ? x1[i + 2] * f1 : 0.0f),
                                             fmaf(x0[i + 3], f0, theirs ? x1[i + 3] * f1 : 0.0f));
                // the fused launch's merge reads the partial soon: keep it in L2
                if (FUSED) st_keep(dst + 4 + c0 + i, v);
                else *reinterpret_cast<float4 *>(dst + 4 + c0 + i) = v;
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (mine) mbar_arrive(&sm.o_empty[0]);
            if (mine1) mbar_arrive(&sm.o_empty[1]);
            mbar_arrive(&sm.pub_empty);
          }
          if (mine) ++uses;
          // (reference max of l and O, sum, visible count, true max)
          if (valid_row) {
            const float4 hd = make_float4(mr, fmaf(lsum, f0, o1.y * f1), (float)nvis + o1.z, fmaxf(m_true, o1.w));
            if (FUSED) st_keep(dst, hd);
            else *reinterpret_cast<float4 *>(dst) = hd;
          }
          if (FUSED) signal_add(&L.a_done[slice_of(L, a)], lane);  // this warp's rows of the partial are written
        }
        ++n_it;
        it += ntile;
      }
    }
  } else if (SUMS) {
    // ------------------------------------------------------------ page sums, norms (warps 12..15)
    // Per tile, one thread per token: the bound of |v|; then, one thread per
    // probe row (TMEM lane) as in the softmax: walks the sums of eight
    // columns that the softmax left in shared memory, cuts them at the page
    // starts and ends (a cut inside a group reads the group's P from tensor
    // memory) and writes log2 of the row's sum over every piece of a page.
    // Here, not in the softmax: there the same work lay on every tile's
    // chain (flash pass 39.8 -> 57.3 ms on 64 layers of 128K tokens and 512
    // probe rows).
    regs_dec<88>();
    const int wq = warp & 3, row = wq * 32 + lane;
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    uint32_t it = 0;
    bool ok = true;
    for (int item = cta; item < n_items && ok; item += ncta) {
      const ItemA a = decode_a(L, item);
      const TcTraj &tr = L.t[a.t];
      const int t0 = a.c * L.chunk_len, t1 = min(tr.S, t0 + L.chunk_len);
      const int ntile = (t1 - t0 + BT - 1) / BT;
      __half *norms = tr.pr.vnorm + (int64_t)(a.li * L.H + a.kvh) * ((tr.S + BT - 1) / BT * BT) + t0 + row;
      __half *piece_row =
          tr.pr.pieces + (int64_t)((a.li * L.H + a.kvh) * tr.nrt + a.rt) * tr.pr.npiece * BM + row;
      const int2 *tiles = tr.pr.tile + t0 / BT;
      const uint2 *cuts = tr.pr.cuts + t0 / 32;
      const bool warp_rows = a.rt * BM + wq * 32 < L.g * tr.W;  // the warp has a probe row of the slice
#pragma unroll 1
      for (int j = 0; j < ntile; ++j) {
        const uint32_t g = it + j;
        const int s2 = g % NVB, b = g & 1;
        const int2 tile = __ldg(&tiles[j]);
        const uint2 cut4 = __ldg(&cuts[4 * j + (lane & 3)]);  // lane i: chunk i mod 4
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.v_full[s2], (g / NVB) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        if (a.rt == 0) norms[j * BT] = norm_bound(sm.v[s2], row);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.v_empty[s2]);
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.p_full[b], (g >> 1) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (!warp_rows) {
          if (lane == 0) mbar_arrive(&sm.s_empty[b]);
          continue;
        }
        __half *dst = piece_row + (int64_t)tile.x * BM;
        const float mu = sm.mused[b][row];
        // run: the row's sum before the chunk; base: before the segment being
        // walked; part: the part of base that comes from a cut group.  A sum
        // of P is within 2^-16 of its terms' sum, a difference of two running
        // sums within 2^-21 of the larger: added on top.
        float run = 0.0f, base = 0.0f, part = 0.0f;
        auto put = [&](float end, float end_part) {
          const float s = fmaxf(end - base, 0.0f) + fmaf(end, 5e-7f, (end_part + part) * 2e-5f);
          *dst = __float2half_ru(fast_log2(s) + mu);
          dst += BM;
        };
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          const float4 gs = sm.gs[b][c][row];
          uint32_t m = __shfl_sync(0xffffffffu, cut4.x, c);
          const uint32_t ends = __shfl_sync(0xffffffffu, cut4.y, c);
#pragma unroll 1
          while (m) {
            const int at = __ffs(m) - 1, q = at >> 3, k = at & 7;
            m &= m - 1;
            float p = 0.0f;
            if (k) {
              uint32_t hi[4], lo[4];
              const uint32_t col = tm + lane_base + b * PW + 16 * NP * c + 4 * q;  // the first two terms of P
              tmem_ld4(col, hi);
              tmem_ld4(col + 16, lo);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 7; ++e) {
                const uint32_t h = hi[e >> 1], w = lo[e >> 1];
                const float x = e & 1 ? __uint_as_float(h & 0xffff0000u) + __uint_as_float(w & 0xffff0000u)
                                      : __uint_as_float(h << 16) + __uint_as_float(w << 16);
                p += e < k ? x : 0.0f;
              }
            }
            const float end = run + (q > 0 ? gs.x : 0.0f) + (q > 1 ? gs.y : 0.0f) + (q > 2 ? gs.z : 0.0f) + p;
            if ((ends >> at) & 1u) put(end, p);
            base = end;
            part = p;
          }
          run += (gs.x + gs.y) + (gs.z + gs.w);
        }
        if (tile.y) put(run, 0.0f);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.s_empty[b]);
      }
      it += ntile;
    }
  } else if (FUSED) {
    // ------------------------------------------------------------ merge (warps 12..15, fused launch only)
    // For each item of this CTA, once every item of its slice has written
    // its partials, the four warps merge this item's share of the slice's
    // probe rows into the row statistics (m, l, n, o); the page-pass CTAs
    // wait for all shares of a slice.  No tensor memory, no TMA.
    regs_dec<48>();
    const int w = warp - 12;
    for (int item = cta; item < n_items; item += ncta) {
      const ItemA a = decode_a(L, item);
      const TcTraj &tr = L.t[a.t];
      const int s = slice_of(L, a), nis = items_per_slice(L, a.t);
      if (!warp_poll_geq(&L.a_done[s], 4u * nis, abort_flag, hdr)) break;
      const int rows = L.g * tr.W, jin = a.c * tr.nrt + a.rt;
      const int r0 = (int)((int64_t)jin * rows / nis), r1 = (int)((int64_t)(jin + 1) * rows / nis);
      for (int row = r0 + w; row < r1; row += 4) merge_row<FUSED>(L, a.t, a.li, a.kvh, row, lane);
      signal_add(&L.merged[s], lane);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tm, 512);
  if (threadIdx.x == 0 && sm.abort_flag) {
    if (FUSED) atomicExch(&hdr->abort, 1);
    record_error(hdr, COMMITKV_ERR_TIMEOUT, 10);
  }
}

template <bool SUMS>
__global__ void __launch_bounds__(SUMS ? 512 : 384, 1) pass_a_tc(const __grid_constant__ TcLaunch L, WsHeader *hdr) {
  extern __shared__ uint8_t smem_raw[];
  flash_body<false, SUMS>(L, hdr, smem_raw, blockIdx.x, gridDim.x);
}


// ============================================================== combine
// Merges the 2 x nchunk partials of one probe row of a (trajectory, layer,
// KV head) slice into its row stats (m, l, n, o): one warp, four channels
// per lane (with 64 channels the upper lanes hold none).
template <bool FUSED>
__device__ __forceinline__ void merge_row(const TcLaunch &L, int t, int li, int kvh, int row, int lane) {
  const TcTraj &tr = L.t[t];
  const int l = L.layer_ids[li];
  const int rt = row / BM, rl = row % BM;
  // partial k = chunk k (one per item: the two softmax warpgroups' states
  // are merged in the CTA)
  auto part = [&](int k) {
    const int item = L.item_off_a[t] + ((li * L.H + kvh) * tr.nchunk + k) * tr.nrt + rt;
    return part_ptr<FUSED>(L, item, 0, rl);
  };
  const int nparts = tr.nchunk;  // at most 32 (checked on the host)
  // headers, one partial per lane: (reference max, sum, visible count, true max)
  const float4 h0 = lane < nparts ? ld_once(part(lane)) : make_float4(-INFINITY, 0.f, 0.f, -INFINITY);
  const float4 h1 = lane + 32 < nparts ? ld_once(part(lane + 32)) : make_float4(-INFINITY, 0.f, 0.f, -INFINITY);
  // the first kBatch partials' outputs, four channels per lane, loaded
  // before the weights are known (the loads depend on nothing)
  constexpr int kBatch = FUSED ? 2 : 8;  // the fused launch's merge warps run on 48 registers
  float4 vb[kBatch];
#pragma unroll
  for (int u = 0; u < kBatch; ++u) vb[u] = u < nparts && lane * 4 < D ? ld_once(part(u) + 4 + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  const float m = warp_max(fmaxf(h0.w, h1.w));  // true row max over the partials (base 2)
  // weight of each partial; a partial that saw nothing (reference -inf) has
  // weight 0 and an unwritten output
  const float a0 = h0.x == -INFINITY ? 0.0f : exp2f(h0.x - m);
  const float a1 = h1.x == -INFINITY ? 0.0f : exp2f(h1.x - m);
  const float lsum = warp_sum(fmaf(h0.y, a0, h1.y * a1));
  const float n = warp_sum(h0.z + h1.z);
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  // outputs, partials in order, in batches whose loads are issued
  // together
  for (int k0 = 0; k0 < nparts; k0 += kBatch) {
    if (k0 > 0) {
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        vb[u] = k0 + u < nparts && lane * 4 < D ? ld_once(part(k0 + u) + 4 + lane * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int k = k0 + u;
      const float a = __shfl_sync(0xffffffffu, k < 32 ? a0 : a1, k & 31);
      if (k >= nparts) break;
      float4 v = vb[u];
      if (a == 0.0f) v = make_float4(0.f, 0.f, 0.f, 0.f);
      o.x = fmaf(v.x, a, o.x);
      o.y = fmaf(v.y, a, o.y);
      o.z = fmaf(v.z, a, o.z);
      o.w = fmaf(v.w, a, o.w);
    }
  }
  const float inv = lsum > 0.0f ? 1.0f / lsum : 0.0f;
  const int h = kvh * L.g + row / tr.W, w = row % tr.W;
  float *dst = tr.stats + (((int64_t)l * L.Hq + h) * tr.W + w) * (D + 4);
  if (lane == 0)
    *reinterpret_cast<float4 *>(dst) = make_float4(m == -INFINITY ? m : m * 0.69314718055994531f, lsum, n, 0.0f);
  const float4 on = make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
  if (lane * 4 < D) *reinterpret_cast<float4 *>(dst + 4 + lane * 4) = on;
  if (!FUSED && L.prune) {  // the terms of bound_kernel; the max as the page pass reads it back
    const float n2 = warp_sum(fmaf(on.x, on.x, fmaf(on.y, on.y, fmaf(on.z, on.z, on.w * on.w))));
    if (lane == 0)
      tr.pr.aux[((int64_t)(li * L.H + kvh) * tr.nrt + rt) * BM + rl] =
          make_float4(m == -INFINITY ? m : (m * 0.69314718055994531f) * 1.4426950408889634f, lsum, sqrtf(n2), 0.0f);
  }
}

// One warp per probe row of the selected layers (the two-launch path).  Four
// blocks a SM: two registers above 64 a thread leave three (36,864 rows of
// 16 chunks: 35 us, 30 so).
__global__ void __launch_bounds__(256, 4) combine_tc(const __grid_constant__ TcLaunch L) {
  const int gw = (blockIdx.x * 256 + threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (gw >= L.row_off[L.n_traj]) return;
  const int t = traj_of(L.row_off, L.n_traj, gw);
  const TcTraj &tr = L.t[t];
  int local = gw - L.row_off[t];
  const int rows = L.g * tr.W;
  const int row = local % rows;
  local /= rows;
  merge_row<false>(L, t, local / L.H, local % L.H, row, lane);
}

// ============================================================== prep
// Per trajectory, once per call:
//   slot_off[E] = sum over F < E of ceil(len_F / 16), slot_off[P] = total
//   (a page that fails the table checks gets no slot and an error is recorded;
//   the pages with slots are disjoint, which bounds the tables);
//   slot_tab[slot] = {first token, valid tokens, page, first/last flags} for
//   every 16-token slot;
//   the pass-B work items: item k takes the pages whose first slot lies in
//   [k * slots_per_item, (k + 1) * slots_per_item);
//   vis_all = number of leading resident tokens visible to every probe row
//   (positions increase, so this is a prefix); nvis_w[w] = number of resident
//   tokens visible to window position w.
// R is cleared, for the atomic maxima that follow.
// For a pruned launch also where the flash pass cuts its row sums (cuts,
// tile, piece_off: a page with slots has one piece per 128-token tile that it
// touches), and the counters of the list passes cleared.
__global__ void __launch_bounds__(1024) prep_kernel(const __grid_constant__ TcLaunch L, WsHeader *hdr) {
  const TcTraj &tr = L.t[blockIdx.x];
  int lane = threadIdx.x % 32, wid = threadIdx.x / 32;
  // one scan gives both the slot offsets (low 32 bits) and the piece offsets
  // (high 32 bits)
  __shared__ unsigned long long s_w[32], s_b;
  __shared__ int s_end[32], s_bend;  // largest end of the pages seen so far
  if (threadIdx.x == 0) s_b = 0ull, s_bend = 0;
  for (int i = threadIdx.x; i < tr.P; i += 1024) tr.R[i] = 0.0f;
  const bool prune = L.prune != 0 && tr.S > 0 && tr.W > 0;
  if (prune) {
    const int ntile = (tr.S + BT - 1) / BT;
    for (int i = threadIdx.x; i < 4 * ntile; i += 1024) tr.pr.cuts[i] = make_uint2(0u, 0u);
    for (int i = threadIdx.x; i < ntile; i += 1024) tr.pr.tile[i] = make_int2(0x7fffffff, 0);
  }
  if (blockIdx.x == 0 && threadIdx.x < 2) hdr->list_work[threadIdx.x] = 0ull;
  __syncthreads();
  for (int c0 = 0; c0 < tr.P; c0 += 1024) {
    int E = c0 + threadIdx.x;
    int ns = 0, ps = 0, pl = 0, end_incl = 0;
    bool span = false;
    if (E < tr.P) {
      ps = tr.ps[E];
      pl = tr.pl[E];
      span = pl >= 0 && ps >= 0 && ps <= tr.S - pl;
      end_incl = span ? ps + pl : 0;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end_incl, o);
      if (lane >= o) end_incl = max(end_incl, y);
    }
    if (lane == 31) s_end[wid] = end_incl;
    __syncthreads();
    int end_before = __shfl_up_sync(0xffffffffu, end_incl, 1);
    if (lane == 0) end_before = 0;
    for (int w = 0; w < wid; ++w) end_before = max(end_before, s_end[w]);
    end_before = max(end_before, s_bend);
    if (E < tr.P) {
      const bool bad = !span || ps < end_before;
      if (bad) record_error(hdr, COMMITKV_ERR_DEVICE_INPUT, E);
      ns = bad ? 0 : (pl + SLOT - 1) / SLOT;
    }
    const int np = ns > 0 ? (ps + pl - 1) / BT - ps / BT + 1 : 0;
    const unsigned long long v = ((unsigned long long)np << 32) | (unsigned)ns;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    if (wid == 0) {
      unsigned long long w = s_w[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      s_w[lane] = w;
    }
    __syncthreads();
    const unsigned long long excl = s_b + (wid ? s_w[wid - 1] : 0ull) + x - v;
    if (E < tr.P) {
      const int off = (int)(excl & 0xffffffffull), piece = (int)(excl >> 32);
      tr.slot_off[E] = off;
      for (int sub = 0; sub < ns; ++sub)
        tr.slot_tab[off + sub] = make_int4(ps + sub * SLOT, min(SLOT, pl - sub * SLOT), E,
                                           (sub == 0 ? 1 : 0) | (sub + 1 == ns ? 2 : 0));
      if (prune) tr.pr.piece_off[E] = piece;
      if (prune && np > 0) {
        const int end = ps + pl;
        atomicOr(&tr.pr.cuts[ps / 32].x, 1u << (ps % 32));
        if (end % BT) {
          atomicOr(&tr.pr.cuts[end / 32].x, 1u << (end % 32));
          atomicOr(&tr.pr.cuts[end / 32].y, 1u << (end % 32));
        }
        for (int k = 0; k < np; ++k) {
          atomicMin(&tr.pr.tile[ps / BT + k].x, piece + k);
          if (k + 1 < np || end % BT == 0) tr.pr.tile[ps / BT + k].y = 1;
        }
      }
    }
    __syncthreads();
    if (threadIdx.x == 1023) s_b += s_w[31], s_bend = max(end_before, end_incl);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int nslot = (int)(s_b & 0xffffffffull);
    tr.slot_off[tr.P] = nslot;
    tr.prep->nitem = (nslot + L.slots_per_item - 1) / L.slots_per_item;
    if (prune) tr.pr.piece_off[tr.P] = (int)(s_b >> 32);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < tr.nbitem; k += 1024) {
    int lo = k * L.slots_per_item, hi = lo + L.slots_per_item;
    int a = 0, b = tr.P;
    while (a < b) {
      int mid = (a + b) >> 1;
      if (tr.slot_off[mid] < lo) a = mid + 1;
      else b = mid;
    }
    int E0 = a;
    b = tr.P;
    while (a < b) {
      int mid = (a + b) >> 1;
      if (tr.slot_off[mid] < hi) a = mid + 1;
      else b = mid;
    }
    int E1 = a;
    int slot0 = E0 < tr.P ? tr.slot_off[E0] : 0;
    int nslot = E1 > E0 ? tr.slot_off[E1] - slot0 : 0;
    int npages = 0;
    for (int E = E0; E < E1; ++E) npages += tr.slot_off[E + 1] > tr.slot_off[E];
    tr.items[2 * k] = make_int4(E0, E1, slot0, nslot);
    tr.items[2 * k + 1] = make_int4(npages, 0, 0, 0);
  }
  for (int w = threadIdx.x; w < tr.W; w += blockDim.x) {
    const int qp = tr.qpos[w];
    int a = 0, b = tr.S;
    while (a < b) {
      int mid = (a + b) >> 1;
      if (tr.pos[mid] <= qp) a = mid + 1;
      else b = mid;
    }
    tr.nvis_w[w] = a;
  }
  if (threadIdx.x == 0) {
    int qmin = 0x7fffffff;
    for (int w = 0; w < tr.W; ++w) qmin = min(qmin, tr.qpos[w]);
    int a = 0, b = tr.S;  // first token with pos > qmin
    while (a < b) {
      int mid = (a + b) >> 1;
      if (tr.pos[mid] <= qmin) a = mid + 1;
      else b = mid;
    }
    tr.prep->vis_all = a;
  }
}

// Work items of the page pass, from the number of slots that the pages really
// have.  The host knows an upper bound only; with items counted from it the
// empty ones fell on some CTAs more than on others (page pass of 36 layers of
// 26.5K tokens 1,855 us, 990 us with the real counts).
struct ItemCount {
  int off[kMaxTc + 1];  // prefix per trajectory
  int per[kMaxTc];      // items per unit
};
// Called by all 32 lanes of one warp.
__device__ __forceinline__ void count_items(const TcLaunch &L, ItemCount &c) {
  const int lane = threadIdx.x % 32;
  int per = 0, n = 0;
  if (lane < L.n_traj) {
    const TcTraj &tr = L.t[lane];
    if (L.item_off_b[lane + 1] > L.item_off_b[lane]) {
      per = tr.prep->nitem;
      n = per * L.n_layers * L.H * tr.nrt;
    }
    c.per[lane] = per;
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, n, o);
    if (lane >= o) n += y;
  }
  if (lane == 0) c.off[0] = 0;
  if (lane < L.n_traj) c.off[lane + 1] = n;
}
static_assert(kMaxTc <= 32, "one lane per trajectory");

// ============================================================== pass B
// TMEM columns: S/P buffers at 0 and PW (as in pass A), page accumulators
// U[0] at 2 PW and U[1] at 2 PW + D.
struct SlotMeta {
  int tok0;   // first resident index of the slot
  int nv;     // valid tokens in the slot (0 for an empty slot)
  int po;     // page ordinal within the CTA's page stream (-1: empty slot)
  int flags;  // bit 0: first slot of its page, bit 1: last slot of its page
};

struct SmemB {
  alignas(1024) uint8_t q[kTileBytes];
  alignas(1024) uint8_t k[NKB][kTileBytes];
  alignas(1024) uint8_t v[NVB][kTileBytes];
  SlotMeta meta[NKB][SLOTS];
  int page_of[NKB][SLOTS];  // page id of each slot
  uint32_t tile_bytes[NKB]; // bytes of the tile's K (and V) copies
  int tile_full[NKB];       // every slot of the tile lies in the prefix all probe rows see
  int pos[4][BT];           // per softmax warp: positions of the current tile
  float fifo_s[NFIFO][BM];  // per page: S_E of every row
  int fifo_n[NFIFO][BM];    // per page: visible count of every row
  int fifo_page[NFIFO];
  ItemCount ic;
  uint64_t q_full, q_empty, k_full[NKB], k_empty[NKB], meta_empty[NKB], v_full[NVB], v_empty[NVB], s_full[2],
      s_empty[2], p_full[2], acc_full[2], acc_empty[2], fifo_full[NFIFO], fifo_empty[NFIFO], drain[2], drain2;
  uint32_t tmem;
  int abort_flag;
};

struct ItemB {
  int t, l, kvh, rt, li;
  int npages;          // pages of the item (with slots)
  int nslot;           // slots of those pages
  const int4 *stab;    // their slot records, or the whole table with
  const int32_t *ids;  // the records' indices (LIST)
};

// LIST: the item is a run of a unit's slot list (pass 0 or 1 of the pruned
// page pass); otherwise a run of consecutive pages.
template <bool LIST>
__device__ __forceinline__ ItemB decode_b(const TcLaunch &L, const ItemCount &ic, int item) {
  ItemB b;
  if constexpr (LIST) {
    const int4 e = L.list_items[item];
    b.t = traj_of(L.unit_off, L.n_traj, e.x);
    const TcTraj &tr = L.t[b.t];
    int local = e.x - L.unit_off[b.t];
    b.ids = tr.pr.list + (int64_t)local * tr.pr.cap + e.y;
    b.stab = tr.slot_tab;
    b.rt = local % tr.nrt;
    local /= tr.nrt;
    b.kvh = local % L.H;
    b.li = local / L.H;
    b.nslot = e.z;
    b.npages = e.w;
  } else {
    b.t = traj_of(ic.off, L.n_traj, item);
    const TcTraj &tr = L.t[b.t];
    int local = item - ic.off[b.t];
    b.rt = local % tr.nrt;
    local /= tr.nrt;
    const int k = local % ic.per[b.t];
    local /= ic.per[b.t];
    b.kvh = local % L.H;
    b.li = local / L.H;
    const int4 e = tr.items[2 * k];
    b.stab = tr.slot_tab + e.z;
    b.ids = nullptr;
    b.nslot = e.w;
    b.npages = tr.items[2 * k + 1].x;
  }
  b.l = L.layer_ids[b.li];
  return b;
}

template <bool FUSED, bool LIST>
__device__ __forceinline__ void page_body(const TcLaunch &L, WsHeader *hdr, uint8_t *smem_raw, const int cta,
                                          const int ncta, const int n_list) {
  SmemB &sm = *reinterpret_cast<SmemB *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  volatile int *abort_flag = &sm.abort_flag;

  if (threadIdx.x == 0) {
    sm.abort_flag = 0;
    mbar_init(&sm.q_full, 1);
    mbar_init(&sm.q_empty, 1);
    for (int s = 0; s < NKB; ++s) {
      mbar_init(&sm.k_full[s], 1);
      mbar_init(&sm.k_empty[s], 1);
      mbar_init(&sm.meta_empty[s], 6);  // four softmax warps and the two P V threads
    }
    for (int s = 0; s < NVB; ++s) {
      mbar_init(&sm.v_full[s], 1);
      mbar_init(&sm.v_empty[s], 2);  // both P V threads
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.s_full[b], 1);
      mbar_init(&sm.s_empty[b], 2);  // both P V threads
      mbar_init(&sm.acc_full[b], 1);
      mbar_init(&sm.acc_empty[b], 4);  // the epilogue warpgroup of that page parity
    }
    // one per S/P buffer: the softmax can finish tile g + 1 before the P V
    // thread has seen tile g, but not tile g + 2, so a parity wait on a
    // per-buffer barrier cannot miss a phase
    mbar_init(&sm.p_full[0], 4);
    mbar_init(&sm.p_full[1], 4);
    for (int f = 0; f < NFIFO; ++f) {
      mbar_init(&sm.fifo_full[f], 4);
      mbar_init(&sm.fifo_empty[f], 4);
    }
    mbar_init(&sm.drain[0], 1);
    mbar_init(&sm.drain[1], 1);
    mbar_init(&sm.drain2, 1);
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem, 512);
    tmem_relinquish();
  }
  if (!LIST && warp == 2) count_items(L, sm.ic);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = sm.tmem;
  // read where it is compared: held in a register by every role it cost
  // spills (the full page pass of 36 layers of 18K tokens, in a register and
  // so, us: pages of 32 tokens 884 and 872, of 100 and 250 784 and 777, of 16
  // 1,408 and 1,417)
  const volatile int *count = &sm.ic.off[L.n_traj];
  auto n_items = [&]() { return LIST ? n_list : *count; };

  // warpgroup 0: TMA producer, two P V issuers (warps 1 and 3), Q K^T issuer; 1: softmax;
  // 2 and 3: epilogue.  Each branch first sets its warpgroup's register
  // budget: 64 + 112 + 2 x 168 per thread = the launch's 4 x 128, with 64
  // channels (a shorter o, more terms of P) 64 + 128 + 2 x 160 (a budget
  // below 128 is set with a decrease, above it with an increase).
  if (warp < 4) {
    regs_dec<64>();
    if (warp == 0) {
      // ------------------------------------------------------------ TMA producer
      // The whole warp works each tile: lanes 0..7 take one 16-token slot each
      // from the slot table, write the tile's slot table to shared memory and
      // issue the copies of the runs of slots that start at them.
      uint64_t pol = policy_evict_first();
      uint32_t it = 0, n_local = 0, n_k = 0, n_v = 0;  // tiles; Q, K and V copies issued
      int po_next = 0;  // page ordinal of the next page to start
      bool stop = false;
      for (int item = cta; item < n_items() && !stop; item += ncta) {
        if (*abort_flag) break;
        ItemB bi = decode_b<LIST>(L, sm.ic, item);
        if (bi.nslot == 0) continue;
        const TcTraj &tr = L.t[bi.t];
        const TcMaps &mp = L.maps[bi.t];
        const int vis_all = tr.prep->vis_all;
        if (n_local > 0 && !__all_sync(0xffffffffu, mbar_wait(&sm.q_empty, (n_local - 1) & 1, kWait, abort_flag))) {
          stop = true;
          break;
        }
        if (lane == 0) {
          mbar_expect_tx(&sm.q_full, kTileBytes);
          int qrow = (bi.l * L.Hq + bi.kvh * L.g) * tr.W + bi.rt * BM;
          tma_q(sm.q, &mp.q, qrow, &sm.q_full, pol);
        }
        ++n_local;
        // Copies of the runs of slots whose rows are contiguous in memory (full
        // slots of one event): a lane that starts a run issues its boxes of 16,
        // 32, 64 or 128 rows.  Called by the whole warp; lanes 0..7 carry a slot.
        auto issue_runs = [&](int tok0, int nv, bool valid, uint8_t *dst, const CUtensorMap *big,
                              const CUtensorMap *small, uint64_t *bar) {
          unsigned vmask = __ballot_sync(0xffffffffu, valid);
          int ptok = __shfl_up_sync(0xffffffffu, tok0, 1), pnv = __shfl_up_sync(0xffffffffu, nv, 1);
          bool pvalid = lane > 0 && ((vmask >> (lane - 1)) & 1u);
          bool start = valid && (!pvalid || pnv != SLOT || ptok + SLOT != tok0);
          unsigned smask = __ballot_sync(0xffffffffu, start);
          if (start) {
            unsigned ends = (smask | ~vmask) & ~((2u << lane) - 1u);  // run boundaries after this lane
            int run = (__ffs(ends) - 1) - lane;                        // lanes >= 8 are never valid
            int done = 0;
            while (done < run) {
              int rem = run - done;
              int lg = rem >= 8 ? 3 : rem >= 4 ? 2 : rem >= 2 ? 1 : 0;
              if (lg == 3 && (lane + done) != 0) lg = 2;  // a 128-row box covers the whole tile
              int tok = tok0 + done * SLOT;
              uint8_t *d = dst + (lane + done) * SLOT * 128;
              const CUtensorMap *m = lg == 3 ? big : small + lg;
              tma4_all(d, m, tok, bi.kvh, bi.l, bar, pol);
              done += 1 << lg;
            }
          }
        };
        // K of tile g (and its slot table) once Q K^T of tile g - NKB is done and
        // its slot table released
        auto load_k = [&](uint32_t g, int j) -> bool {
          int s3 = g % NKB;
          bool w_ok = g < NKB || (mbar_wait(&sm.k_empty[s3], ((g / NKB) - 1) & 1, kWait, abort_flag) &&
                                  mbar_wait(&sm.meta_empty[s3], ((g / NKB) - 1) & 1, kWait, abort_flag));
          if (!__all_sync(0xffffffffu, w_ok)) return false;
          int sl = j * SLOTS + lane;
          bool valid = lane < SLOTS && sl < bi.nslot;
          int4 rec = valid ? bi.stab[LIST ? bi.ids[sl] : sl] : make_int4(0, 0, -1, 0);
          const unsigned starts = __ballot_sync(0xffffffffu, valid && (rec.w & 1));
          SlotMeta mt;
          mt.tok0 = rec.x;
          mt.nv = valid ? rec.y : 0;
          mt.po = valid ? po_next + __popc(starts & ((2u << lane) - 1u)) - 1 : -1;
          mt.flags = valid ? rec.w & 3 : 0;
          po_next += __popc(starts);
          if (lane < SLOTS) {
            sm.meta[s3][lane] = mt;
            sm.page_of[s3][lane] = rec.z;
          }
          const bool tfull = __all_sync(0xffffffffu, !valid || rec.x + rec.y <= vis_all);
          const uint32_t bytes = __popc(__ballot_sync(0xffffffffu, valid)) * (uint32_t)NH * SLOT * 128u;
          __syncwarp();  // the slot table is written before the arrival that publishes it
          if (lane == 0) {
            sm.tile_bytes[s3] = bytes;
            sm.tile_full[s3] = tfull;
            mbar_expect_tx(&sm.k_full[s3], bytes);
          }
          __syncwarp();
          issue_runs(mt.tok0, mt.nv, valid, sm.k[s3], &mp.k, mp.kb, &sm.k_full[s3]);
          ++n_k;
          return true;
        };
        // V of tile g once P V of tile g - NVB is done
        auto load_v = [&](uint32_t g) -> bool {
          int s3 = g % NKB, s2 = g % NVB;
          bool w_ok = g < NVB || mbar_wait(&sm.v_empty[s2], ((g / NVB) - 1) & 1, kWait, abort_flag);
          if (!__all_sync(0xffffffffu, w_ok)) return false;
          SlotMeta mt = sm.meta[s3][lane < SLOTS ? lane : 0];
          bool valid = lane < SLOTS && mt.po >= 0;
          if (lane == 0) mbar_expect_tx(&sm.v_full[s2], sm.tile_bytes[s3]);
          __syncwarp();
          issue_runs(mt.tok0, mt.nv, valid, sm.v[s2], &mp.v, mp.vb, &sm.v_full[s2]);
          ++n_v;
          return true;
        };
        // K runs one tile ahead of V
        int ntile = (bi.nslot + SLOTS - 1) / SLOTS;
        stop = !load_k(it, 0);
        for (int j = 0; j < ntile && !stop; ++j) {
          if (j + 1 < ntile && !load_k(it + j + 1, j + 1)) stop = true;
          else if (!load_v(it + j)) stop = true;
        }
        it += ntile;
      }
      if (lane == 0 && *abort_flag) {
        // let the copies already issued land before the CTA leaves
        for (uint32_t u = (n_k > NKB ? n_k - NKB : 0); u < n_k; ++u)
          mbar_wait_drain(&sm.k_full[u % NKB], (u / NKB) & 1, kWait);
        for (uint32_t u = (n_v > NVB ? n_v - NVB : 0); u < n_v; ++u)
          mbar_wait_drain(&sm.v_full[u % NVB], (u / NVB) & 1, kWait);
        if (n_local > 0) mbar_wait_drain(&sm.q_full, (n_local - 1) & 1, kWait);
      }
    } else if (warp == 1 || warp == 3) {
      // ------------------------------------------------------------ P V issuers
      // Two issuing threads, one per page accumulator: warp 1 the even page
      // ordinals (U[0]), warp 3 the odd ones (U[1]).  Both release the S/P
      // buffer, the V stage and the slot table of every tile.
      const int par = warp == 1 ? 0 : 1;
      if (lane == 0) {
        uint32_t it = 0;
        bool ok = true;
        for (int item = cta; item < n_items() && ok; item += ncta) {
          ItemB bi = decode_b<LIST>(L, sm.ic, item);
          if (bi.nslot == 0) continue;
          int ntile = (bi.nslot + SLOTS - 1) / SLOTS;
          for (int j = 0; j < ntile && ok; ++j) {
            uint32_t g = it + j;
            int s3 = g % NKB, s2 = g % NVB, b = g & 1;
            if (!mbar_wait(&sm.p_full[b], (g >> 1) & 1, kWait, abort_flag) ||
                !mbar_wait(&sm.v_full[s2], (g / NVB) & 1, kWait, abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll 1
            for (int q = 0; q < SLOTS && ok; ++q) {
              SlotMeta mt = sm.meta[s3][q];
              if (mt.po < 0 || (mt.po & 1) != par) continue;
              const int a = par;
              if ((mt.flags & 1) && mt.po >= 2) {
                if (!mbar_wait(&sm.acc_empty[a], ((mt.po >> 1) - 1) & 1, kWait, abort_flag)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
              }
              issue_pv_step(tm, 2 * PW + a * D, sm.v[s2], b, q, (mt.flags & 1) != 0);
              if (mt.flags & 2) mma_commit(&sm.acc_full[a]);
            }
            mma_commit(&sm.s_empty[b]);
            mma_commit(&sm.v_empty[s2]);
            mbar_arrive(&sm.meta_empty[s3]);  // done with the slot table
          }
          it += ntile;
        }
        if (*abort_flag) {
          mma_commit(&sm.drain[par]);  // every MMA issued by this thread has completed
          mbar_wait_drain(&sm.drain[par], 0, kWait);
        }
      }
    } else if (warp == 2) {
      // ------------------------------------------------------------ Q K^T issuer
      // A second issuing thread: S = Q K^T of tile g needs only its K copy and
      // the S/P buffer that P V of tile g - 2 has finished reading.
      if (lane == 0) {
        uint32_t it = 0, n_local = 0;
        bool ok = true;
        for (int item = cta; item < n_items() && ok; item += ncta) {
          ItemB bi = decode_b<LIST>(L, sm.ic, item);
          if (bi.nslot == 0) continue;
          int ntile = (bi.nslot + SLOTS - 1) / SLOTS;
          if (!mbar_wait(&sm.q_full, n_local & 1, kWait, abort_flag)) break;
          ++n_local;
          tc_fence_after();
          for (int j = 0; j < ntile && ok; ++j) {
            uint32_t g = it + j;
            int s3 = g % NKB, b = g & 1;
            if (!mbar_wait(&sm.k_full[s3], (g / NKB) & 1, kWait, abort_flag) ||
                (g >= 2 && !mbar_wait(&sm.s_empty[b], ((g >> 1) - 1) & 1, kWait, abort_flag))) {
              ok = false;
              break;
            }
            tc_fence_after();
            issue_qk(tm, sm.q, sm.k[s3], b);
            mma_commit(&sm.s_full[b]);
            mma_commit(&sm.k_empty[s3]);
            if (j + 1 == ntile) mma_commit(&sm.q_empty);  // every Q K^T of this item is issued
          }
          it += ntile;
        }
        if (*abort_flag) {
          mma_commit(&sm.drain2);  // every MMA issued by this thread has completed
          mbar_wait_drain(&sm.drain2, 0, kWait);
        }
      }
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------ softmax (warps 4..7)
    if constexpr (D == 128) regs_dec<112>();  // below the launch's 128: a decrease
    const int wq = warp & 3;
    const int row = wq * 32 + lane;
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    uint32_t it = 0;
    int po_seen = 0;
    float S_cur = 0.0f;
    int n_cur = 0;
    bool ok = true;
    for (int item = cta; item < n_items() && ok; item += ncta) {
      ItemB bi = decode_b<LIST>(L, sm.ic, item);
      if (bi.nslot == 0) continue;
      const TcTraj &tr = L.t[bi.t];
      int rows = L.g * tr.W;
      int grow = bi.rt * BM + row;
      bool valid_row = grow < rows;
      const bool warp_rows = grow - lane < rows;  // a warp without a row of the slice only keeps the pages' order
      int qp = -0x7fffffff;
      // the row stats of this slice are complete once every share is merged
      if (FUSED && !warp_poll_geq(&L.merged[slice_of(L, bi)], 4u * items_per_slice(L, bi.t), abort_flag, hdr)) {
        ok = false;
        break;
      }
      // rows outside the slice, or rows that see nothing, get e = 0 everywhere
      float neg_m2 = -INFINITY;
      if (valid_row) {
        int h = bi.kvh * L.g + grow / tr.W, w = grow % tr.W;
        qp = tr.qpos[w];
        float mn = tr.stats[(((int64_t)bi.l * L.Hq + h) * tr.W + w) * (D + 4)];
        if (mn != -INFINITY) neg_m2 = -mn * 1.4426950408889634f;
      }
      int ntile = (bi.nslot + SLOTS - 1) / SLOTS;
      for (int j = 0; j < ntile && ok; ++j) {
        uint32_t g = it + j;
        int s = g % NKB, b = g & 1;
        // the slot table of this stage is published with its K copies (warp-
        // uniform results keep the lanes together for the collective ops)
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.k_full[s], (g / NKB) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        // slots inside the prefix every probe row sees need no position test
        const bool full = sm.tile_full[s] != 0;
        if (!full) {  // each warp keeps its own copy: no cross-warp barrier
          __syncwarp();
#pragma unroll 1
          for (int c = lane; c < BT; c += 32) {
            const SlotMeta mt = sm.meta[s][c / SLOT];
            int i = c % SLOT;
            sm.pos[wq][c] = i < mt.nv ? tr.pos[mt.tok0 + i] : 0x7fffffff;
          }
          __syncwarp();
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[b], (g >> 1) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        // Per 32-column chunk (two slots): e = exp(s - m) on the visible page
        // tokens (a visibility bit mask turns the others into -inf, so e = 0);
        // P as the (hi, lo) bf16 pair written over the S columns just read;
        // slot sums accumulate into page sums S_E, which go to the page FIFO
        // when the page's last slot is done.  The chunk loop is not unrolled:
        // a small loop body keeps the instruction cache warm.
        const int po_first = po_seen;
#pragma unroll 1
        for (int ch = 0; ch < BT / 32 && ok; ++ch) {
          const SlotMeta m0 = sm.meta[s][2 * ch], m1 = sm.meta[s][2 * ch + 1];
          uint32_t vm = (m0.nv >= SLOT ? 0xffffu : (1u << max(m0.nv, 0)) - 1u) |
                        ((m1.nv >= SLOT ? 0xffffu : (1u << max(m1.nv, 0)) - 1u) << 16);
          float s0 = 0.0f, s1 = 0.0f;
          if (warp_rows) {
            float x[32];
            // tensor-memory loads and stores are warp-collective: the lanes
            // may have left the bounded waits above on different iterations
            __syncwarp();
            tmem_ld32f(tm + lane_base + b * PW + S0 + 32 * ch, x);
            if (!full) {
#pragma unroll 1
              for (int i = 0; i < 32; ++i)
                if (sm.pos[wq][32 * ch + i] > qp) vm &= ~(1u << i);
            }
            if (!valid_row) vm = 0;
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) x[i] = (vm >> i) & 1u ? x[i] : -INFINITY;
#pragma unroll
            for (int i = 0; i < 32; i += 2)
              exp2_pair(&x[i], make_float2(L.scale_log2, L.scale_log2), make_float2(neg_m2, neg_m2));
            s0 = sum8(x) + sum8(x + 8);
            s1 = sum8(x + 16) + sum8(x + 24);
            store_p(tm + lane_base + b * PW, ch, x);
          }
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const SlotMeta mt = h2 ? m1 : m0;
            if (mt.po < 0) continue;
            if (mt.flags & 1) {
              S_cur = 0.0f;
              n_cur = 0;
            }
            S_cur += h2 ? s1 : s0;
            n_cur += __popc(h2 ? vm >> 16 : vm & 0xffffu);
            if (mt.flags & 2) {
              int f = po_seen % NFIFO;
              if (!__all_sync(0xffffffffu, po_seen < NFIFO || mbar_wait(&sm.fifo_empty[f], ((po_seen / NFIFO) - 1) & 1,
                                                                           kWait, abort_flag))) {
                ok = false;
                break;
              }
              sm.fifo_s[f][row] = S_cur;
              sm.fifo_n[f][row] = n_cur;
              if (row == 0) sm.fifo_page[f] = sm.page_of[s][2 * ch + h2];
              ++po_seen;
            }
          }
        }
        __syncwarp();
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&sm.p_full[b]);
          // publish the pages this tile finished to the epilogue
          for (int k = po_first; k < po_seen; ++k) mbar_arrive(&sm.fifo_full[k % NFIFO]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.meta_empty[s]);  // done with the slot table
      }
      it += ntile;
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 8..15)
    // The two warpgroups take alternate pages: warpgroup 2 the even page
    // ordinals (accumulator U[0]), warpgroup 3 the odd ones (U[1]).  Each
    // thread owns one row and all 128 channels of that row's output o.
    regs_inc<D == 128 ? 168 : 160>();
    const int wq = warp & 3;
    const int par = (warp - 8) >> 2;
    const int row = wq * 32 + lane;
    const uint32_t lane_base = (uint32_t)(wq * 32) << 16;
    const uint32_t u_col = 2 * PW + par * D;
    int po = 0;
    bool ok = true;
    for (int item = cta; item < n_items() && ok; item += ncta) {
      ItemB bi = decode_b<LIST>(L, sm.ic, item);
      if (bi.nslot == 0) continue;
      const TcTraj &tr = L.t[bi.t];
      int rows = L.g * tr.W;
      int grow = bi.rt * BM + row;
      bool valid_row = grow < rows;
      const bool warp_rows = grow - lane < rows;
      int h = bi.kvh * L.g + (valid_row ? grow / tr.W : 0), w = valid_row ? grow % tr.W : 0;
      if (FUSED && !warp_poll_geq(&L.merged[slice_of(L, bi)], 4u * items_per_slice(L, bi.t), abort_flag, hdr)) {
        ok = false;
        break;
      }
      float2 o2[D / 2];
      float lsum = 0.0f, onorm = 0.0f;
      int nvis = 0;
      {
        const float *st = tr.stats + (((int64_t)bi.l * L.Hq + h) * tr.W + w) * (D + 4);
        float4 hd = valid_row ? *reinterpret_cast<const float4 *>(st) : make_float4(0.f, 0.f, 0.f, 0.f);
        lsum = hd.y;
        nvis = valid_row ? tr.nvis_w[w] : 0;
        float ss = 0.0f;
#pragma unroll
        for (int c = 0; c < D; c += 4) {
          float4 v = valid_row ? *reinterpret_cast<const float4 *>(st + 4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
          // explicit FMAs: the same rounding in every kernel this body is compiled into
          ss = fmaf(v.x, v.x, ss);
          ss = fmaf(v.y, v.y, ss);
          ss = fmaf(v.z, v.z, ss);
          ss = fmaf(v.w, v.w, ss);
          o2[c / 2] = make_float2(v.x, v.y);
          o2[c / 2 + 1] = make_float2(v.z, v.w);
        }
        onorm = sqrtf(ss);
      }
      for (int k = 0; k < bi.npages && ok; ++k, ++po) {
        if ((po & 1) != par) continue;
        int f = po % NFIFO;
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.fifo_full[f], (po / NFIFO) & 1, kWait, abort_flag) &&
                                         mbar_wait(&sm.acc_full[par], (po >> 1) & 1, kWait, abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        float S_E = sm.fifo_s[f][row];
        int n_E = sm.fifo_n[f][row];
        int E = sm.fifo_page[f];
        const float2 nS = make_float2(-S_E, -S_E);
        // ||U_E - S_E o||^2 over 16-column pieces of U_E
        float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
        if (!warp_rows) {  // no row of the slice: only hands the accumulator back
          if (lane == 0) {
            mbar_arrive(&sm.acc_empty[par]);
            mbar_arrive(&sm.fifo_empty[f]);
          }
          continue;
        }
#pragma unroll
        for (int c0 = 0; c0 < D; c0 += 16) {
          uint32_t r[16];
          tmem_ld16(tm + lane_base + u_col + c0, r);
          tmem_wait_ld();
          if (c0 + 16 == D) {  // U_E is in registers: hand the accumulator back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              mbar_arrive(&sm.acc_empty[par]);
              mbar_arrive(&sm.fifo_empty[f]);
            }
          }
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            float2 d0 = ffma2(nS, o2[(c0 + i) / 2], make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])));
            float2 d1 = ffma2(nS, o2[(c0 + i) / 2 + 1], make_float2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])));
            acc0 = ffma2(d0, d0, acc0);
            acc1 = ffma2(d1, d1, acc1);
          }
        }
        float num2 = (acc0.x + acc0.y) + (acc1.x + acc1.y);
        float r = valid_row ? effect_value(n_E, nvis, S_E, lsum, num2, onorm) : 0.0f;
        if (valid_row && tr.headR) atomic_max_nonneg(tr.headR + ((int64_t)bi.l * L.Hq + h) * tr.P + E, r);
        float rm = r;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) rm = fmaxf(rm, __shfl_xor_sync(0xffffffffu, rm, off));
        if (lane == 0) atomic_max_nonneg(tr.R + E, rm);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tm, 512);
  if (threadIdx.x == 0 && sm.abort_flag) {
    if (FUSED) atomicExch(&hdr->abort, 1);
    record_error(hdr, COMMITKV_ERR_TIMEOUT, 11);
  }
}

__global__ void __launch_bounds__(512, 1) pass_b_tc(const __grid_constant__ TcLaunch L, WsHeader *hdr) {
  extern __shared__ uint8_t smem_raw[];
  page_body<false, false>(L, hdr, smem_raw, blockIdx.x, gridDim.x, 0);
}

// The page pass over the units' slot lists (list pass `which`).
__global__ void __launch_bounds__(512, 1) pass_b_list_tc(const __grid_constant__ TcLaunch L, WsHeader *hdr, int which) {
  extern __shared__ uint8_t smem_raw[];
  const int n = (int)(hdr->list_work[which] & 0xffffffffull);
  if ((int)blockIdx.x >= n) return;
  page_body<false, true>(L, hdr, smem_raw, blockIdx.x, gridDim.x, n);
}

// ============================================================== bounds and lists
// R(E) is a maximum over units and rows (Eq. 7), so a unit whose effects
// cannot exceed a value of R(E) that is already there need not score page E.
// With s the page's share of the row's attention,
//   r = ||U_E - S_E o|| / ((l - S_E) ||o||)  <=  s / (1 - s) (1 + max|v| / ||o||)
// since ||U_E|| <= S_E max|v|.  The flash pass leaves log2 S_E (rounded up)
// of every row and page and |v| of every token; this kernel takes the
// maximum of the bound over the unit's rows, its 128 less those past the
// slice's end: the flash pass writes nothing for those, and the workspace
// holds what was there (36 layers of 1.9K + 0.5K tokens, 32 rows a unit, with
// NaN there: 675 us a call, 386 so).  Shares above 0.9, where
// rounding in l - S_E matters, rows with an output norm that is not an
// ordinary number, and NaN give an infinite bound; the factors cover the
// rounding of the terms.
constexpr int kBoundPages = 64;  // pages per block: eight consecutive ones per warp
__global__ void __launch_bounds__(256) bound_kernel(const __grid_constant__ TcLaunch L) {
  const int t = traj_of(L.bound_off, L.n_traj, blockIdx.x);
  const TcTraj &tr = L.t[t];
  const TcPrune &pr = tr.pr;
  const int npb = (tr.P + kBoundPages - 1) / kBoundPages, local = blockIdx.x - L.bound_off[t];
  const int unit = local / npb, rt = unit % tr.nrt, slice = unit / tr.nrt;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  constexpr int kPer = kBoundPages / 8;
  const int Ew = local % npb * kBoundPages + warp * kPer, np = min(kPer, tr.P - Ew);
  if (np <= 0) return;
  const __half *pieces = pr.pieces + (int64_t)unit * pr.npiece * BM + 4 * lane;  // lane i: rows 4 i .. 4 i + 3
  const __half *vn = pr.vnorm + (int64_t)slice * ((tr.S + BT - 1) / BT * BT);
  // rows of this lane that the unit has: the others' pieces are not read
  const int rows = min(4, L.g * tr.W - rt * BM - 4 * lane);
  const uint2 none = make_uint2(0xfc00fc00u, 0xfc00fc00u);  // -inf: no mass
  auto load = [&](int piece) {
    return rows > 0 ? __ldg(reinterpret_cast<const uint2 *>(pieces + (int64_t)piece * BM)) : none;
  };
  // lane i reads page i's table entries; the loads of all pages are issued
  // before any is used
  const int po_l = pr.piece_off[Ew + min(lane, np)];
  const int ps_l = tr.ps[Ew + min(lane, np - 1)], pl_l = tr.pl[Ew + min(lane, np - 1)];
  uint2 w0[kPer], w1[kPer];
  unsigned short v0[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int p0 = __shfl_sync(0xffffffffu, po_l, i), p1 = __shfl_sync(0xffffffffu, po_l, i + 1);
    const int b = __shfl_sync(0xffffffffu, ps_l, i), n = __shfl_sync(0xffffffffu, pl_l, i);
    const bool any = i < np && p1 > p0;
    w0[i] = any ? load(p0) : none;
    w1[i] = any && p1 > p0 + 1 ? load(p0 + 1) : none;
    v0[i] = any && lane < n ? __half_as_ushort(vn[b + lane]) : (unsigned short)0;
  }
  // share of a row = 2^(L - ref), L the piece's log2 (P and the page's own sum
  // differ by rounding: 0.002 and 1e-6 |max| on top); dead rows have share 0
  float ref[4], inv_o[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 a = k < rows ? pr.aux[(int64_t)unit * BM + 4 * lane + k] : make_float4(-INFINITY, 0.0f, 1.0f, 0.0f);
    const bool live = a.x != -INFINITY;  // the row sees something
    ref[k] = live ? a.x - (4e-3f + 1e-6f * fabsf(a.x)) + fast_log2(a.y) : INFINITY;
    inv_o[k] = !live ? 0.0f : a.z > 1e-15f && a.z < 1e30f ? 1.01f / a.z : INFINITY;
  }
  auto add = [&](float (&S)[4], uint2 w) {
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&w.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&w.y));
    S[0] += fast_exp2(a.x - ref[0]);
    S[1] += fast_exp2(a.y - ref[1]);
    S[2] += fast_exp2(b.x - ref[2]);
    S[3] += fast_exp2(b.y - ref[3]);
  };
  unsigned mine = 0;  // lane i: the bound of page i
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int p0 = __shfl_sync(0xffffffffu, po_l, i), p1 = __shfl_sync(0xffffffffu, po_l, i + 1);
    const int b = __shfl_sync(0xffffffffu, ps_l, i), n = __shfl_sync(0xffffffffu, pl_l, i);
    unsigned vb = v0[i];
    float S[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    add(S, w0[i]);
    if (i < np && p1 > p0) {
      if (p1 > p0 + 1) add(S, w1[i]);
      // pages of more than 32 tokens, or more than two tiles
      for (int k = lane + 32; k < n; k += 32) vb = max(vb, (unsigned)__half_as_ushort(vn[b + k]));
      for (int p = p0 + 2; p < p1; ++p) add(S, load(p));
    }
    const float v = __half2float(__ushort_as_half((unsigned short)__reduce_max_sync(0xffffffffu, vb)));
    unsigned mx = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float r = __fdividef(S[k], 1.0f - S[k]) * fmaf(v, inv_o[k], 1.0f);
      const unsigned rb = S[k] < 0.9f ? __float_as_uint(r) & 0x7fffffffu : 0x7f800000u;  // a NaN stays above every bound
      mx = max(mx, k < rows ? rb : 0u);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == i) mine = mx;
  }
  if (lane < np) pr.bound[(int64_t)unit * tr.P + Ew + lane] = __uint_as_float(mine);
}

// Per page the unit with the largest bound: a block takes 32 pages, its
// warps the units in turn.
__global__ void __launch_bounds__(512) seed_kernel(const __grid_constant__ TcLaunch L) {
  const int t = traj_of(L.seed_off, L.n_traj, blockIdx.x);
  const TcTraj &tr = L.t[t];
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int E = (blockIdx.x - L.seed_off[t]) * 32 + lane, units = L.unit_off[t + 1] - L.unit_off[t];
  __shared__ unsigned long long s_key[16][32];
  unsigned long long key = 0ull;
  if (E < tr.P && tr.slot_off[E + 1] > tr.slot_off[E])
    for (int u = warp; u < units; u += 16) {
      const unsigned b = __float_as_uint(tr.pr.bound[(int64_t)u * tr.P + E]);  // non-negative, infinite or NaN
      const unsigned long long k = ((unsigned long long)b << 32) | (unsigned)u;
      if (b != 0u && k > key) key = k;
    }
  s_key[warp][lane] = key;
  __syncthreads();
  if (warp == 0 && E < tr.P) {
    for (int w = 1; w < 16; ++w) key = key > s_key[w][lane] ? key : s_key[w][lane];
    tr.pr.seed[E] = key;
  }
}

// Writes the slot list of one unit per block and its work items.  Pass 0
// takes the pages whose seed this unit is; pass 1, when R holds the seeds'
// effects, the other pages whose bound is above R, or infinite: then the
// effect may be a NaN, which the maximum ranks above an infinite R.  A page
// whose bound is 0 has no visible mass and effect 0.  Items: item k of a unit takes the pages
// whose first slot in its list lies in [k n, (k + 1) n).  A unit that keeps half
// of the slots or more takes twice as many an item, as the full page pass does,
// where that leaves kPairedPerSm items a SM: every item costs its start.
// Nothing dropped, 36 layers of 18K tokens (2,592 such items) in pages of 100
// and 250: page pass 833 us, 784 so, and in pages of 16 1,495 and 1,443;
// with 576 items a call takes longer (2.4K tokens, 32 rows: 431 us, 469 to 585
// paired; 16 layers of 64 channels, 9.2K: 613 and 660), and so does one whose
// units keep little (all paired, 16K + 2K with a sixth kept: page pass 248 us, 298).
constexpr int kPairedPerSm = 8;
constexpr int kMaxBuckets = 1024;
__global__ void __launch_bounds__(256) list_kernel(const __grid_constant__ TcLaunch L, WsHeader *hdr, int which, int sm_count) {
  const int t = traj_of(L.unit_off, L.n_traj, blockIdx.x);
  const TcTraj &tr = L.t[t];
  const TcPrune &pr = tr.pr;
  const int unit = blockIdx.x - L.unit_off[t];
  const int per = max(kListSlotsPerItem, (pr.cap + kMaxBuckets - 1) / kMaxBuckets);
  const int nbuckets = (pr.cap + per - 1) / per;
  __shared__ unsigned long long s_first[kMaxBuckets];  // {first list entry, first page} of every bucket
  __shared__ unsigned long long s_warp[8], s_run;
  __shared__ int s_n, s_at;
  for (int i = threadIdx.x; i < nbuckets; i += 256) s_first[i] = ~0ull;
  if (threadIdx.x == 0) s_run = 0ull, s_n = 0;
  __syncthreads();
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  int32_t *list = pr.list + (int64_t)unit * pr.cap;
  for (int c0 = 0; c0 < tr.P; c0 += 256) {
    const int E = c0 + threadIdx.x;
    bool take = false;
    int s0 = 0, ns = 0;
    if (E < tr.P) {
      s0 = tr.slot_off[E];
      ns = tr.slot_off[E + 1] - s0;
      const bool mine = pr.seed[E] != 0ull && (unsigned)(pr.seed[E] & 0xffffffffull) == (unsigned)unit;
      if (which == 0) take = mine;
      else {
        const float b = pr.bound[(int64_t)unit * tr.P + E];
        take = !mine && b != 0.0f && (!(b <= tr.R[E]) || b == INFINITY);
      }
      take = take && ns > 0;
    }
    // running (slots, pages taken) before this page
    const unsigned long long v = take ? ((unsigned long long)1 << 32) | (unsigned)ns : 0ull;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    unsigned long long excl = s_run + x - v, total = 0ull;
    for (int w = 0; w < 8; ++w) {
      if (w < warp) excl += s_warp[w];
      total += s_warp[w];
    }
    if (take) {
      const int off = (int)(excl & 0xffffffffull), page = (int)(excl >> 32);
      for (int k = 0; k < ns; ++k) list[off + k] = s0 + k;
      atomicMin(&s_first[off / per], ((unsigned long long)off << 32) | (unsigned)page);
    }
    __syncthreads();
    if (threadIdx.x == 0) s_run += total;
    __syncthreads();
  }
  const unsigned long long all = ((s_run & 0xffffffffull) << 32) | (s_run >> 32);  // {slots, pages}
  const int64_t slots = tr.slot_off[tr.P];
  if (2 * (int64_t)(s_run & 0xffffffffull) >= slots &&
      gridDim.x * slots >= (int64_t)kPairedPerSm * sm_count * 2 * kListSlotsPerItem) {
    for (int i = 2 * threadIdx.x; i + 1 < nbuckets; i += 512) {  // the smaller entry: the earlier pages
      s_first[i] = min(s_first[i], s_first[i + 1]);
      s_first[i + 1] = ~0ull;
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < nbuckets; i += 256)
    if (s_first[i] != ~0ull) atomicAdd(&s_n, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    // {pages, items} of the unit in one addition
    s_at = s_n ? (int)(atomicAdd(&hdr->list_work[which], (s_run & ~0xffffffffull) | (unsigned)s_n) & 0xffffffffull) : 0;
    s_n = 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbuckets; i += 256) {
    const unsigned long long a = s_first[i];
    if (a == ~0ull) continue;
    unsigned long long e = all;
    for (int j = i + 1; j < nbuckets; ++j)
      if (s_first[j] != ~0ull) {
        e = s_first[j];
        break;
      }
    const int off = (int)(a >> 32), nslot = (int)(e >> 32) - off;
    const int npages = (int)(e & 0xffffffffull) - (int)(a & 0xffffffffull);
    L.list_items[s_at + atomicAdd(&s_n, 1)] = make_int4((int)blockIdx.x, off, nslot, npages);
  }
}

#if CKV_TC_D == 128
// ============================================================== fused
// One cooperative launch over all SMs: CTAs [0, n_a) run the flash pass
// (and merge the row stats slice by slice), CTAs [n_a, grid) run the page
// pass, each page-pass item waiting until its slice's stats are merged.
// Items of both passes are taken in slice order, so the page pass re-reads
// a slice's keys and values shortly after the flash pass read them, while
// they are still in L2.  Every cross-CTA wait is bounded.
__global__ void __launch_bounds__(512, 1) score_fused_tc(const __grid_constant__ TcLaunch L, WsHeader *hdr) {
  extern __shared__ uint8_t smem_raw[];
  if ((int)blockIdx.x < L.n_a) flash_body<true, false>(L, hdr, smem_raw, blockIdx.x, L.n_a);
  else page_body<true, false>(L, hdr, smem_raw, blockIdx.x - L.n_a, gridDim.x - L.n_a, 0);
}
#endif

// ============================================================== host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

bool map_q(CUtensorMap *m, const void *q, uint64_t rows) {
  auto enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)D, rows};
  cuuint64_t strides[1] = {(cuuint64_t)D * 2};
  cuuint32_t box[2] = {64, BM};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(q), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool map_kv(CUtensorMap *m, const void *base, int S, int H, int M, int64_t st, int64_t sh, int64_t sl,
            int box_rows) {
  auto enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)(S > 0 ? S : 1), (cuuint64_t)H, (cuuint64_t)M};
  cuuint64_t strides[3] = {(cuuint64_t)st * 2, (cuuint64_t)sh * 2, (cuuint64_t)sl * 2};
  cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

static size_t smem_a() { return sizeof(SmemA) + 1024; }
static size_t smem_b() { return sizeof(SmemB) + 1024; }

bool build_maps(TcMaps &mp, const TrajDev &t, int M, int H, int Hq) {
  uint64_t qrows = (uint64_t)M * Hq * (uint64_t)(t.W > 0 ? t.W : 1);
  bool ok = map_q(&mp.q, t.q, qrows) && map_kv(&mp.k, t.k, t.S, H, M, t.st, t.sh, t.sl, BT) &&
            map_kv(&mp.v, t.v, t.S, H, M, t.st, t.sh, t.sl, BT);
  for (int i = 0; i < 3 && ok; ++i)
    ok = map_kv(&mp.kb[i], t.k, t.S, H, M, t.st, t.sh, t.sl, SLOT << i) &&
         map_kv(&mp.vb[i], t.v, t.S, H, M, t.st, t.sh, t.sl, SLOT << i);
  return ok;
}

cudaError_t launch_score_tc(TcLaunch &L, WsHeader *hdr, cudaStream_t s, int sm_count) {
  cudaError_t e;
  for (int t = 0; t < L.n_traj; ++t)
    if (L.t[t].nchunk > 32) return cudaErrorInvalidValue;  // the row merge takes at most 64 partials
  const int na_items = L.from_stats ? 0 : L.item_off_a[L.n_traj];
  const int nb_items = L.item_off_b[L.n_traj];
#if CKV_TC_D == 128
  if (L.fused && na_items > 0) {
    // fused: prep, then one cooperative launch of both passes
    const size_t smem = smem_a() > smem_b() ? smem_a() : smem_b();
    e = cudaFuncSetAttribute(score_fused_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, score_fused_tc, 512, smem);
    if (e != cudaSuccess) return e;
    if (per_sm != 1) return cudaErrorInvalidConfiguration;  // one CTA per SM: all 512 TMEM columns each
    L.n_a = fused_flash_ctas(L, sm_count);
    int nb = sm_count - L.n_a;
    nb = nb < nb_items ? nb : nb_items;
    if (nb < 1 && nb_items > 0) return cudaErrorInvalidConfiguration;
    prep_kernel<<<L.n_traj, 1024, 0, s>>>(L, hdr);
    launch_count() += 2;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemsetAsync(L.a_done, 0, (size_t)L.slice_off[L.n_traj] * kCounterStride * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(L.merged, 0, (size_t)L.slice_off[L.n_traj] * kCounterStride * 4, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&hdr->abort, 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&L, (void *)&hdr};
    return cudaLaunchCooperativeKernel((const void *)score_fused_tc, dim3(L.n_a + nb), dim3(512), args, smem, s);
  }
#endif
  const auto pass_a = L.prune ? pass_a_tc<true> : pass_a_tc<false>;
  e = cudaFuncSetAttribute(pass_a, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_a());
  if (e != cudaSuccess) return e;
  e = L.prune ? cudaFuncSetAttribute(pass_b_list_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b())
              : cudaFuncSetAttribute(pass_b_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b());
  if (e != cudaSuccess) return e;
  if (L.prune) {
    L.bound_off[0] = L.seed_off[0] = 0;
    for (int t = 0; t < L.n_traj; ++t) {
      const int units = L.unit_off[t + 1] - L.unit_off[t], P = units > 0 ? L.t[t].P : 0;
      L.bound_off[t + 1] = L.bound_off[t] + units * ((P + kBoundPages - 1) / kBoundPages);
      L.seed_off[t + 1] = L.seed_off[t] + (P + 31) / 32;
    }
  }
  prep_kernel<<<L.n_traj, 1024, 0, s>>>(L, hdr);
  launch_count() += 1 + (na_items > 0);
  if (na_items > 0) pass_a<<<na_items < sm_count ? na_items : sm_count, L.prune ? 512 : 384, smem_a(), s>>>(L, hdr);
  const int rows = L.from_stats ? 0 : L.row_off[L.n_traj];
  if (rows > 0) combine_tc<<<(rows * 32 + 255) / 256, 256, 0, s>>>(L);
  launch_count() += rows > 0;
  if (L.prune) {
    launch_count() += 6;
    const int units = L.unit_off[L.n_traj];
    bound_kernel<<<L.bound_off[L.n_traj], 256, 0, s>>>(L);
    seed_kernel<<<L.seed_off[L.n_traj], 512, 0, s>>>(L);
    for (int which = 0; which < 2; ++which) {
      list_kernel<<<units, 256, 0, s>>>(L, hdr, which, sm_count);
      pass_b_list_tc<<<sm_count, 512, smem_b(), s>>>(L, hdr, which);
    }
    return cudaGetLastError();
  }
  if (nb_items > 0) pass_b_tc<<<nb_items < sm_count ? nb_items : sm_count, 512, smem_b(), s>>>(L, hdr);
  launch_count() += nb_items > 0;
  return cudaGetLastError();
}

}  // namespace CKV_TC_NS
}  // namespace tc
}  // namespace ckv
