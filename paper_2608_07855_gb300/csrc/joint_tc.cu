// Greedy joint test (Section 3.3, Eq. 11) on the 5th-generation tensor
// cores: bf16 K/V/Q, head_dim 128, fp32 accumulation in tensor memory.
//
// One cooperative persistent kernel, one CTA of 256 threads per SM.  A
// group is 128 probe rows of one (trajectory, selected layer, KV head), TMEM
// lane i holding row i; the CTA's threads form two teams of four warps, and
// thread i of each team works on row i: the teams split the pages in the
// softmax and the channels in the epilogue.  In every round (joint_common.cuh) a
// group makes up to two passes of the same machinery over a list of at
// most four pages:
//   fold  the pages of the previous round that were accepted: their D_E are
//         computed again (bit-identical to the values that round used) and
//         added, in candidate order, into the row's D_A, S_A, n_A in the
//         workspace;
//   scan  the round's candidates: Eq. 6 on A u T for every non-empty subset
//         T of them, max over the rows (Eq. 7) into the round's table.
// A pass stages Q (once per group and round) and the pages' K and V rows in
// shared memory (cp.async into the 128-byte-swizzled layout) and issues
//   S = Q K^T       one MMA chain with N = 32 x pages, TMEM columns 256..383
//   e = exp(s - m)  per row on the page's visible tokens (m = the row's
//                   final max); S_E = sum e, n_E = count; P = e written
//                   over S as a bf16 (hi, lo) pair
//   U_E = P V_E     per page and 64-channel half, TMEM columns 64 c, TS form
//                   (P from tensor memory, V from shared memory)
// and the epilogue reads U_E 8 columns at a time (o and D_A of the channel
// half staged in shared memory while the MMAs run): D_E = U_E - S_E o.  In
// the scan the sums of the subsets are built as a tree in which every
// subset adds its largest page last, so each is the sum that the
// one-page-at-a-time scan forms, ((D_A + D_b1) + D_b2) + ... + D_c, and its
// squared norm accumulates over the channels in order.
// Pages longer than 32 tokens are taken in 32-token chunks: U accumulates
// over the chunks, and the chunks' QK and softmax are redone for the second
// channel half.  Every mbarrier wait is bounded (1 s); on expiry the kernel
// records COMMITKV_ERR_TIMEOUT, raises the abort flag that the grid barrier
// watches, waits (bounded) for its MMAs in flight, frees its tensor memory
// and returns.
//
// What bounds it: the chain of a block's two groups per round (95 candidates
// of 36 layers of 20K tokens, 802 us: 24 rounds of two groups in 69K cycles;
// of these the epilogue's packed FMAs 30 %, staging 15 %, the P V waits and
// softmax 13 % each, the grid barrier with its stragglers 10 %, Eq. 6 and the
// plan 15 %).  Neither memory (6 %) nor the tensor cores are near a limit.
#include "joint_common.cuh"
#include "sm103.cuh"

namespace ckv {
namespace {

using namespace ckv::sm103;
using joint::kCombos;
using joint::kRound;

constexpr int D = 128;
constexpr int kRows = 128;   // probe rows per group (MMA M, TMEM lanes)
constexpr int kCT = 32;      // page tokens per chunk (the QK N of one page)
constexpr int kTeam = 128;                 // threads per team (one per row)
constexpr int kThreads = 2 * kTeam;
constexpr uint64_t kWait = 1000000000ull;
constexpr uint32_t kQHalf = kRows * 128;         // one 64-channel half of the Q tile: 16 KB
constexpr uint32_t kKHalf = kRound * kCT * 128;  // K rows of all pages, one half: 16 KB
constexpr uint32_t kVHalf = kCT * 128;           // V rows of one page, one half: 4 KB
constexpr uint32_t kColS = 256;                  // TMEM column of page 0's S/P (kCT per page)
constexpr int kHalfPad = 68;                     // floats per row of the o / D_A half buffers
constexpr int kCached = 2;                       // groups per block whose row data stays in shared memory

struct SmemJ {
  alignas(1024) uint8_t q[2 * kQHalf];
  alignas(1024) uint8_t k[2 * kKHalf];
  alignas(1024) uint8_t v[kRound][2 * kVHalf];
  // o and D_A of one 64-channel half of every row (each thread its own
  // row; the padding keeps the rows' 16-byte words in distinct banks)
  alignas(16) float oh[kRows][kHalfPad];
  alignas(16) float dah[kRows][kHalfPad];
  float Sc[kRound][kRows];     // S_E of every page and row (written by the page's team)
  int nc[kRound][kRows];       // n_E
  float part[kCombos + 1][kRows];  // team 1's sums of squares (and ||o||^2) for team 0
  float part2[kCombos / 2 + 1][kRows];  // team 0's, for the subsets that team 1 evaluates
  // the row data of the block's first kCached groups, kept from round to
  // round: final max (base 2), exp-sum, visible count, position, S_A, n_A
  float rc_m2[kCached][kRows], rc_l[kCached][kRows], rc_SA[kCached][kRows];
  int rc_nvis[kCached][kRows], rc_qp[kCached][kRows], rc_nA[kCached][kRows];
  int pos[kRound][kCT];
  // the round's pages of the current group's trajectory: [0] the previous round's accepted
  // pages (to fold), [1] the candidates; {start, length}
  int plan_n[2];
  int2 plan[2][kRound];
  unsigned rmax[16];
  uint64_t bar;       // Q K^T done (one issuing thread)
  uint64_t bar_pv;    // P V done (two issuing threads)
  uint64_t drain[2];  // an issuing thread's MMAs done (after an abort)
  uint32_t tmem;
  int abort_flag;
};

struct Group {
  int t, l, li, kvh, rows, row0;
  // row 0 of the group in Q, the statistics and D_A: the rows of a KV head
  // lie one after another in all three
  const __nv_bfloat16 *q;
  const float *st;
  float *da;
};

// What a thread keeps of its probe row.
struct Row {
  bool ok;          // inside the group
  int64_t grow;     // index into S_A
  float m2, l;      // final max in base-2 units, exp-sum
  int nvis, qp;
  float SA;
  int nA;
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// K-major tile of 128-byte rows in two 64-channel halves half_bytes apart:
// the descriptor of k-step ks (16 channels).
__device__ __forceinline__ uint64_t desc_kmajor(const uint8_t *tile, uint32_t half_bytes, int ks) {
  return smem_desc(smem_addr(tile) + (ks >> 2) * half_bytes + (ks & 3) * 32, 16, 1024, kSwizzle128B);
}
// V rows of one page as the MN-major B operand (k = tokens, n = the 64
// channels of half h): k-step ks (16 tokens).
__device__ __forceinline__ uint64_t desc_v(const uint8_t *tile, int h, int ks) {
  return smem_desc(smem_addr(tile) + h * kVHalf + ks * 2048, kVHalf, 1024, kSwizzle128B);
}
// TMEM column of the 8 packed P columns (hi or lo) of page c, k-step ks.
__device__ __forceinline__ uint32_t p_col(int c, int ks, int lo) {
  return kColS + kCT * c + 32 * (ks >> 1) + 8 * (ks & 1) + 16 * lo;
}
static_assert(kRound * kCT <= kThreads, "one thread per staged position");
static_assert(kCT == 32, "one 32-column TMEM load covers a page chunk's scores");

__device__ __forceinline__ Group decode_group(const JointLaunch &L, int grp) {
  const Batch &b = L.batch;
  Group G;
  G.t = joint::find_group_traj(L.group_off, b.n_traj, grp);
  int local = grp - L.group_off[G.t], nrb = L.nrb[G.t];
  const int rb = local % nrb;
  local /= nrb;
  G.kvh = local % b.H;
  G.li = local / b.H;
  G.l = b.layer_ids[G.li];
  G.rows = b.g * b.t[G.t].W;
  G.row0 = rb * kRows;
  const int64_t row = ((int64_t)G.l * b.Hq + G.kvh * b.g) * b.t[G.t].W + G.row0;
  G.q = static_cast<const __nv_bfloat16 *>(b.t[G.t].q) + row * D;
  G.st = L.stats[G.t] + row * (D + 4);
  G.da = L.DA + (L.row_off[G.t] + (int64_t)(G.li * b.H + G.kvh) * G.rows + G.row0) * D;
  return G;
}

// Waits for the MMAs committed to a pass barrier; uniform over the block.
__device__ __forceinline__ bool wait_mma(SmemJ &s, uint64_t *bar, uint32_t &phase) {
  bool ok = mbar_wait(bar, phase, kWait, &s.abort_flag);
  phase ^= 1u;
  ok = __syncthreads_and(ok) != 0;
  if (ok) tc_fence_after();
  return ok;
}

constexpr int kSub = 8;  // channels per epilogue step

// Starts the copies of o and D_A of the team's 32 channels of half h of the
// warp's 32 rows into those rows of the half buffers, eight lanes to a row's
// 128 bytes (each thread its own row: 32 lines per instruction; 1,117 us
// for the 95 candidates below, 863 so).  The wait for them is followed by a __syncwarp.
__device__ __forceinline__ void stage_half(SmemJ &s, const Group &G, int h) {
  const int lane = threadIdx.x % 32, c0 = 32 * (threadIdx.x / kTeam) + 4 * (lane % 8);
  const int i0 = threadIdx.x % kTeam - lane + lane / 8;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + 4 * u;
    if (G.row0 + i < G.rows) {
      cp_async16(&s.oh[i][c0], G.st + i * (D + 4) + 4 + 64 * h + c0);
      cp_async16(&s.dah[i][c0], G.da + i * D + 64 * h + c0);
    }
  }
}
// The same elements of D_A back to the workspace.
__device__ __forceinline__ void unstage_half(const SmemJ &s, const Group &G, int h) {
  const int lane = threadIdx.x % 32, c0 = 32 * (threadIdx.x / kTeam) + 4 * (lane % 8);
  const int i0 = threadIdx.x % kTeam - lane + lane / 8;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + 4 * u;
    if (G.row0 + i < G.rows)
      *reinterpret_cast<float4 *>(G.da + i * D + 64 * h + c0) = *reinterpret_cast<const float4 *>(&s.dah[i][c0]);
  }
}

// 32 lanes x 8 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[kSub]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// Largest member of the non-empty set T (a constant after unrolling).
__host__ __device__ constexpr int top_bit(int T) { return T >= 8 ? 3 : T >= 4 ? 2 : T >= 2 ? 1 : 0; }

// The round's plan for trajectory t (every group of it in this block uses the
// same): called by the whole block.  Worked out by every thread for every
// group, decision after decision, it lay on each group's chain (95 candidates
// of 36 layers of 20K tokens: 1,199 us, 1,115 so).
__device__ __forceinline__ void make_plan(SmemJ &s, const JointLaunch &L, WsHeader *hdr, int t, int r, int kc) {
  __syncthreads();  // the previous plan has been read
  const TrajDev &tr = L.batch.t[t];
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x, c = lane % kRound, set = lane / kRound;  // lanes 0..3: to fold; 4..7: candidates
    const int kp = r > 0 ? joint::round_count(L, t, r - 1) : 0;
    const int rr = set == 0 ? r - 1 : r, n = set == 0 ? kp : kc;
    // page spans first: they do not depend on the decisions
    int E = -1, ps = 0, pl = 0;
    if (set < 2 && c < n) {
      E = L.cand[t][rr * kRound + c];
      if (E < 0 || E >= tr.P) {
        record_error(hdr, COMMITKV_ERR_DEVICE_INPUT, -4);
      } else {
        ps = tr.ps[E];
        pl = tr.pl[E];
        if (pl < 0 || ps < 0 || ps > tr.S - pl) {
          record_error(hdr, COMMITKV_ERR_DEVICE_INPUT, E);
          ps = pl = 0;
        }
      }
    }
    const unsigned acc = r > 0 ? joint::resolve_round(joint::round_table(L, r - 1) + t * kCombos, kp, L.tau) : 0u;
    if (set == 0 && c < kp && ((acc >> c) & 1u)) s.plan[0][__popc(acc & ((1u << c) - 1u))] = make_int2(ps, pl);
    if (set == 1 && c < kc) s.plan[1][c] = make_int2(ps, pl);
    if (lane == 0) {
      s.plan_n[0] = __popc(acc);
      s.plan_n[1] = kc;
    }
  }
  __syncthreads();
}

// One pass over the pages list[0..n) (n <= kRound).  kScan: accumulates the
// squared norms of the subset sums over the team's channels into ss, and
// o's into on2 (even and odd channels apart); otherwise adds the pages' D_E into D_A in the workspace.
// S_E and n_E of every page are left in Sc and nc.  The fold takes the
// channel halves in the order 1, 0 and leaves o and the new D_A of half 0 in
// the half buffers, where a scan with have_half finds them.  Returns false on
// a timeout.
template <bool kScan>
__device__ __forceinline__ bool run_pass(SmemJ &s, const JointLaunch &L, WsHeader *hdr, const Group &G,
                                         const Row &rw, const int2 *list, int n, bool stage_q, bool have_half, uint32_t tm,
                                         uint32_t lane_base, uint32_t &phase, uint32_t &phase_pv,
                                         float2 (&ss)[kCombos], float2 &on2,
                                         float (&Sc)[kRound], int (&nc)[kRound]) {
  const Batch &b = L.batch;
  const TrajDev &tr = b.t[G.t];
  const int tid = threadIdx.x, team = tid / kTeam, r = tid % kTeam;
  int nch = 1;
#pragma unroll
  for (int c = 0; c < kRound; ++c) {
    Sc[c] = 0.0f;
    nc[c] = 0;
    if (c < n) nch = max(nch, (list[c].y + kCT - 1) / kCT);
  }
  const __nv_bfloat16 *kp =
      static_cast<const __nv_bfloat16 *>(tr.k) + (int64_t)G.l * tr.sl + (int64_t)G.kvh * tr.sh;
  const __nv_bfloat16 *vp =
      static_cast<const __nv_bfloat16 *>(tr.v) + (int64_t)G.l * tr.sl + (int64_t)G.kvh * tr.sh;

  for (int hh = 0; hh < 2; ++hh) {
    const int h = kScan ? hh : 1 - hh;
    for (int j = 0; j < nch; ++j) {
      // tokens of page c in this chunk
      const auto ntok = [&](int c) { return min(kCT, max(0, list[c].y - j * kCT)); };
      if (hh == 0 || nch > 1) {
        // ---- stage (the MMAs that read the buffers have completed)
        __syncthreads();
        // 16 lanes copy a row of 256 bytes, the block 16 rows at a time
        const int k16 = tid & 15, i0 = tid >> 4;
        if (stage_q && hh == 0 && j == 0) {
#pragma unroll
          for (int i = i0; i < kRows; i += kThreads / 16)
            if (G.row0 + i < G.rows)
              cp_async16(s.q + (k16 >> 3) * kQHalf + sw128_offset(i, k16 & 7), G.q + i * D + 8 * k16);
        }
#pragma unroll 1
        for (int c = 0; c < n; ++c) {
          const int nt = ntok(c);
#pragma unroll
          for (int i = i0; i < kCT; i += kThreads / 16)
            if (i < nt) {
              const int64_t off = (int64_t)(list[c].x + j * kCT + i) * tr.st + 8 * k16;
              cp_async16(s.k + (k16 >> 3) * kKHalf + sw128_offset(kCT * c + i, k16 & 7), kp + off);
              cp_async16(s.v[c] + (k16 >> 3) * kVHalf + sw128_offset(i, k16 & 7), vp + off);
            }
        }
        if (tid < n * kCT) {
          const int c = tid / kCT, i = tid % kCT;
          s.pos[c][i] = i < ntok(c) ? tr.pos[list[c].x + j * kCT + i] : 0;
        }
        cp_async_wait_all();
        fence_proxy_async();
        __syncthreads();
        // ---- S = Q K^T for all pages of the pass
        if (tid == 0) {
          tc_fence_after();
          const uint32_t idesc = idesc_bf16_f32(kRows, kCT * n, 0, 0);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks)
            mma_bf16(tm + kColS, desc_kmajor(s.q, kQHalf, ks), desc_kmajor(s.k, kKHalf, ks), idesc, ks > 0);
          mma_commit(&s.bar);
        }
        if (!wait_mma(s, &s.bar, phase)) return false;
        // ---- e = exp(s - m) on the visible tokens; P over S (team t takes
        // the pages c = t mod 2)
#pragma unroll 1
        for (int c = team; c < n; c += 2) {
          float x[32];
          uint32_t pk[32];
          const uint32_t addr = tm + lane_base + kColS + kCT * c;
          tmem_ld32f(addr, x);
          tmem_wait_ld();
          // the chunk's visible tokens: positions increase along the page,
          // so they are a prefix, whole unless the row's position cuts it
          const int nt = ntok(c);
          int ne = 0;
          if (rw.ok && nt > 0) {
            if (s.pos[c][nt - 1] <= rw.qp) {
              ne = nt;
            } else {
#pragma unroll 1
              for (int i = 0; i < nt; ++i) ne += s.pos[c][i] <= rw.qp ? 1 : 0;
            }
          }
          float se = 0.0f;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float e = i < ne ? fast_exp2(fmaf(x[i], b.scale_log2, -rw.m2)) : 0.0f;
            se += e;
            x[i] = e;
          }
          if (hh == 0) {
            s.Sc[c][r] = j == 0 ? se : s.Sc[c][r] + se;
            s.nc[c][r] = j == 0 ? ne : s.nc[c][r] + ne;
          }
          split_pack32(x, pk);
          tmem_st32(addr, pk);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncthreads();
      }
      // ---- U_E (+)= P V_E for channel half h; two threads issue, the even
      // and the odd pages (accumulators of their own), and both commit
      if (tid == 0 || tid == 32) {
        tc_fence_after();
        const uint32_t idesc = idesc_bf16_f32(kRows, 64, 0, 1);
#pragma unroll 1
        for (int c = tid / 32; c < n; c += 2) {
          const int nks = max(1, (ntok(c) + 15) / 16);
#pragma unroll 1
          for (int ks = 0; ks < nks; ++ks) {
            const uint64_t bd = desc_v(s.v[c], h, ks);
            mma_bf16_ts(tm + 64 * c, tm + p_col(c, ks, 0), bd, idesc, (j > 0 || ks > 0) ? 1u : 0u);
            mma_bf16_ts(tm + 64 * c, tm + p_col(c, ks, 1), bd, idesc, 1u);
          }
        }
        mma_commit(&s.bar_pv);
      }
      const bool last = j == nch - 1;
      if (last && !(have_half && h == 0)) stage_half(s, G, h);  // in flight while the MMAs run
      if (!wait_mma(s, &s.bar_pv, phase_pv)) return false;
      if (last) {
        cp_async_wait_all();
        __syncwarp();  // the warp's rows of the half buffers
        if (hh == 0) {
#pragma unroll
          for (int c = 0; c < kRound; ++c)
            if (c < n) {
              Sc[c] = s.Sc[c][r];
              nc[c] = s.nc[c][r];
            }
        }
        // ---- epilogue over the team's 32 channels of half h, kSub at a time
#pragma unroll 1
        for (int q = 4 * team; q < 4 * team + 4; ++q) {
          float o[kSub], da[kSub];
#pragma unroll
          for (int u4 = 0; u4 < kSub / 4; ++u4) {
            const float4 x = *reinterpret_cast<const float4 *>(&s.oh[r][kSub * q + 4 * u4]);
            const float4 y = *reinterpret_cast<const float4 *>(&s.dah[r][kSub * q + 4 * u4]);
            o[4 * u4] = x.x, o[4 * u4 + 1] = x.y, o[4 * u4 + 2] = x.z, o[4 * u4 + 3] = x.w;
            da[4 * u4] = y.x, da[4 * u4 + 1] = y.y, da[4 * u4 + 2] = y.z, da[4 * u4 + 3] = y.w;
          }
          uint32_t u[kRound][kSub];
#pragma unroll
          for (int c = 0; c < kRound; ++c)
            if (c < n) tmem_ld8(tm + lane_base + 64 * c + kSub * q, u[c]);
          tmem_wait_ld();
          // two channels per packed instruction (an addition as a product
          // with 1: the same rounding)
          const float2 one2 = make_float2(1.0f, 1.0f);
#pragma unroll
          for (int i = 0; i < kSub; i += 2) {
            const float2 o2 = make_float2(o[i], o[i + 1]);
            float2 de[kRound];
#pragma unroll
            for (int c = 0; c < kRound; ++c)
              de[c] = c < n ? ffma2(make_float2(-Sc[c], -Sc[c]), o2,
                                    make_float2(__uint_as_float(u[c][i]), __uint_as_float(u[c][i + 1])))
                            : make_float2(0.0f, 0.0f);
            if constexpr (kScan) {
              on2 = ffma2(o2, o2, on2);
              float2 p[1 << kRound];
              // all 15 subsets, also in a pass of fewer pages (their D_E are
              // zero and the sums are not used): with a branch per subset the
              // compiler could not interleave them (863 us, 829 so)
              p[0] = make_float2(da[i], da[i + 1]);
#pragma unroll
              for (int T = 1; T < (1 << kRound); ++T) {
                p[T] = ffma2(de[top_bit(T)], one2, p[T & ~(1 << top_bit(T))]);
                ss[T - 1] = ffma2(p[T], p[T], ss[T - 1]);
              }
            } else {
              float2 x = make_float2(da[i], da[i + 1]);
#pragma unroll
              for (int c = 0; c < kRound; ++c)
                if (c < n) x = ffma2(de[c], one2, x);
              da[i] = x.x;
              da[i + 1] = x.y;
            }
          }
          if constexpr (!kScan) {
            float4 *pa = reinterpret_cast<float4 *>(&s.dah[r][kSub * q]);
#pragma unroll
            for (int u4 = 0; u4 < kSub / 4; ++u4)
              pa[u4] = make_float4(da[4 * u4], da[4 * u4 + 1], da[4 * u4 + 2], da[4 * u4 + 3]);
          }
        }
        if constexpr (!kScan) {
          __syncwarp();
          unstage_half(s, G, h);
          // read again by this block alone (the group stays with it): no
          // fence beyond it, whose wait for the writes lay on every fold (95
          // candidates of 36 layers of 20K tokens: 826 us, 802 so)
          __threadfence_block();
        }
      }
      // the epilogue's TMEM reads are done before the next MMAs write
      tc_fence_before();
      __syncthreads();
    }
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, 1) joint_tc_kernel(const __grid_constant__ JointLaunch L,
                                                             WsHeader *hdr) {
  extern __shared__ uint8_t smem_raw[];
  SmemJ &s = *reinterpret_cast<SmemJ *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const Batch &b = L.batch;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;

  // Rows past a page's end are never written: they keep finite values (zero
  // or an earlier page's), whose scores are masked and whose V rows meet
  // P = 0.
  for (int i = tid; i < (int)(sizeof(s.q) / 16); i += kThreads) reinterpret_cast<uint4 *>(s.q)[i] = uint4{};
  for (int i = tid; i < (int)(sizeof(s.k) / 16); i += kThreads) reinterpret_cast<uint4 *>(s.k)[i] = uint4{};
  for (int i = tid; i < (int)(sizeof(s.v) / 16); i += kThreads) reinterpret_cast<uint4 *>(&s.v[0][0])[i] = uint4{};
  for (int i = tid; i < kRows * kHalfPad; i += kThreads) (&s.oh[0][0])[i] = (&s.dah[0][0])[i] = 0.0f;
  if (tid == 0) {
    s.abort_flag = 0;
    mbar_init(&s.bar, 1);
    mbar_init(&s.bar_pv, 2);
    mbar_init(&s.drain[0], 1);
    mbar_init(&s.drain[1], 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&s.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = s.tmem;
  // warps w and w + 4 (the two teams) reach TMEM lanes 32 (w mod 4) ..
  const uint32_t lane_base = (uint32_t)((warp % 4) * 32) << 16;
  uint32_t phase = 0, phase_pv = 0;
  bool ok = true;

  const int rounds = joint::round_total(L);
  const int ngroups = L.group_off[b.n_traj];
  for (int r = 0; r < rounds && ok; ++r) {
    float *tab_r = joint::round_table(L, r);
    int plan_of = -1;  // trajectory of the plan in shared memory
    for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
      const Group G = decode_group(L, grp);
      const TrajDev &tr = b.t[G.t];
      const int kc = joint::round_count(L, G.t, r);
      if (kc == 0) continue;
      if (plan_of != G.t) {
        make_plan(s, L, hdr, G.t, r, kc);
        plan_of = G.t;
      }
      const int nf = s.plan_n[0];
      const int2 *fold = s.plan[0], *cand = s.plan[1];

      Row rw;
      const int row = G.row0 + tid % kTeam;
      rw.ok = row < G.rows;
      rw.grow = L.row_off[G.t] + (int64_t)(G.li * b.H + G.kvh) * G.rows + (rw.ok ? row : 0);
      const float *st = G.st + (rw.ok ? tid % kTeam : 0) * (D + 4);
      // the block's k-th group; its row data is read from global memory in
      // the first round and from the shared copy after that
      const int kslot = (grp - (int)blockIdx.x) / (int)gridDim.x, rr = tid % kTeam;
      if (kslot < kCached && r > 0) {
        rw.m2 = s.rc_m2[kslot][rr];
        rw.l = s.rc_l[kslot][rr];
        rw.nvis = s.rc_nvis[kslot][rr];
        rw.qp = s.rc_qp[kslot][rr];
        rw.SA = s.rc_SA[kslot][rr];
        rw.nA = s.rc_nA[kslot][rr];
      } else {
        const float mn = rw.ok ? st[0] : -__builtin_huge_valf();
        rw.m2 = mn == -__builtin_huge_valf() ? mn : mn * 1.4426950408889634f;
        rw.l = rw.ok ? st[1] : 0.0f;
        rw.nvis = rw.ok ? (int)st[2] : 0;
        rw.qp = rw.ok ? tr.qpos[row % tr.W] : -0x7fffffff;
        rw.SA = rw.ok ? L.SA[rw.grow * 2] : 0.0f;
        rw.nA = rw.ok ? (int)L.SA[rw.grow * 2 + 1] : 0;
      }
      if (tid < 16) s.rmax[tid] = 0u;

      float2 ss2[kCombos], on2p = make_float2(0.0f, 0.0f);
      float Sc[kRound];
      int nc[kRound];
#pragma unroll
      for (int i = 0; i < kCombos; ++i) ss2[i] = make_float2(0.0f, 0.0f);
      if (nf > 0) {
        if (!run_pass<false>(s, L, hdr, G, rw, fold, nf, true, false, tm, lane_base, phase, phase_pv, ss2, on2p, Sc,
                             nc)) {
          ok = false;
          break;
        }
#pragma unroll
        for (int c = 0; c < kRound; ++c)
          if (c < nf) {
            rw.SA += Sc[c];
            rw.nA += nc[c];
          }
        if (rw.ok && tid < kTeam) {
          L.SA[rw.grow * 2] = rw.SA;
          L.SA[rw.grow * 2 + 1] = (float)rw.nA;
        }
      }
      if (kslot < kCached && tid < kTeam) {  // read again by both teams in the next round
        s.rc_m2[kslot][rr] = rw.m2;
        s.rc_l[kslot][rr] = rw.l;
        s.rc_nvis[kslot][rr] = rw.nvis;
        s.rc_qp[kslot][rr] = rw.qp;
        s.rc_SA[kslot][rr] = rw.SA;
        s.rc_nA[kslot][rr] = rw.nA;
      }
      if (!run_pass<true>(s, L, hdr, G, rw, cand, kc, nf == 0, nf > 0, tm, lane_base, phase, phase_pv, ss2, on2p,
                          Sc, nc)) {
        ok = false;
        break;
      }
      // the channel sums of the thread; team 0 evaluates the subsets
      // T = 1..8 and team 1 the subsets T = 9..15, each with the other team's
      // sums of its channels added (one addition of two floats: the same
      // value in either order)
      constexpr int kSplit = kCombos / 2 + 1;  // subsets T <= kSplit go to team 0
      float ss[kCombos], on2 = on2p.x + on2p.y;
#pragma unroll
      for (int i = 0; i < kCombos; ++i) ss[i] = ss2[i].x + ss2[i].y;
      if (tid >= kTeam) {
#pragma unroll
        for (int i = 0; i < kSplit; ++i) s.part[i][rr] = ss[i];
        s.part[kCombos][rr] = on2;
      } else {
#pragma unroll
        for (int i = kSplit; i < kCombos; ++i) s.part2[i - kSplit][rr] = ss[i];
        s.part2[kCombos - kSplit][rr] = on2;
      }
      __syncthreads();
      {
        // The thread's subsets T0 .. T0 + 7, all values before the first
        // reduction (one subset after another their divisions and roots lay
        // on one chain).
        const bool t1 = tid >= kTeam;
        const float *other = t1 ? &s.part2[0][rr] : &s.part[0][rr];
        const int T0 = t1 ? kSplit + 1 : 1;
        on2 += t1 ? s.part2[kCombos - kSplit][rr] : s.part[kCombos][rr];
        // Eq. 6 on A u T for every non-empty subset T of the round's pages;
        // S and n added in candidate order
        const float onorm = sqrtf(on2);
        float rv[kSplit];
#pragma unroll
        for (int i = 0; i < kSplit; ++i) {
          const int T = T0 + i;
          const float v = (t1 ? (i < kCombos - kSplit ? ss[kSplit + i] : 0.0f) : ss[i]) + other[i * kRows];
          float S_tot = rw.SA;
          int n_tot = rw.nA;
#pragma unroll
          for (int c = 0; c < kRound; ++c)
            if ((T >> c) & 1) {
              S_tot += Sc[c];
              n_tot += nc[c];
            }
          rv[i] = rw.ok ? effect_value(n_tot, rw.nvis, S_tot, rw.l, v, onorm) : 0.0f;
        }
        unsigned mine = 0u;  // lane i: the warp's maximum of subset T0 + i
#pragma unroll
        for (int i = 0; i < kSplit; ++i) {
          const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(rv[i]));
          if (lane == i) mine = mx;
        }
        if (lane < kSplit && T0 + lane < (1 << kc)) atomicMax(&s.rmax[T0 + lane - 1], mine);
      }
      __syncthreads();
      if (tid < (1 << kc) - 1) atomic_max_nonneg(tab_r + G.t * kCombos + tid, __uint_as_float(s.rmax[tid]));
    }
    if (!ok) break;
    if (!joint::grid_barrier(hdr, gridDim.x)) {
      ok = false;
      break;
    }
    if (blockIdx.x == 0) joint::publish_round(L, r);
  }

  if (!ok) {
    // a wait ran out (or another block gave up): leave the grid barrier to
    // the others and let the MMAs in flight finish before the memory goes
    if (tid == 0) {
      if (s.abort_flag) record_error(hdr, COMMITKV_ERR_TIMEOUT, -5);
      atomicExch(&hdr->abort, 1);
    }
    if (tid == 0 || tid == 32) {  // the issuing threads: every MMA of theirs has completed
      mma_commit(&s.drain[tid / 32]);
      mbar_wait_drain(&s.drain[tid / 32], 0, kWait);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

}  // namespace

// bf16, head_dim 128, and 16-byte aligned rows of K, V, Q and the stats.
bool joint_tc_eligible(const JointLaunch &L) {
  const Batch &b = L.batch;
  if (b.dtype != COMMITKV_BF16 || b.d != D) return false;
  for (int t = 0; t < b.n_traj; ++t) {
    const TrajDev &tr = b.t[t];
    if (tr.P == 0 || tr.W == 0) continue;
    if ((reinterpret_cast<uintptr_t>(tr.k) | reinterpret_cast<uintptr_t>(tr.v) |
         reinterpret_cast<uintptr_t>(tr.q) | reinterpret_cast<uintptr_t>(L.stats[t])) & 15)
      return false;
    if ((tr.sl | tr.sh | tr.st) & 7) return false;
  }
  return true;
}

int joint_tc_rows_per_group() { return kRows; }

cudaError_t launch_joint_tc(const JointLaunch &L, WsHeader *hdr, cudaStream_t stream, int sm_count) {
  const size_t smem = sizeof(SmemJ) + 1024;
  cudaError_t e = cudaFuncSetAttribute(joint_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, joint_tc_kernel, kThreads, smem);
  if (e != cudaSuccess) return e;
  // one CTA per SM: each takes all 512 TMEM columns
  if (per_sm != 1) return cudaErrorInvalidConfiguration;
  const int ngroups = L.group_off[L.batch.n_traj];
  const int grid = ngroups < sm_count ? ngroups : sm_count;
  if (grid < 1) return cudaSuccess;
  void *args[] = {(void *)&L, (void *)&hdr};
  ++launch_count();
  return cudaLaunchCooperativeKernel((const void *)joint_tc_kernel, dim3(grid), dim3(kThreads), args, smem,
                                     stream);
}

}  // namespace ckv
