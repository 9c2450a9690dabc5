// Compression checkpoint (Section 3.3, Eq. 12-13) and the shared-index
// gather of keys, values and absolute positions (Eq. 4).
//
// select  a cluster of blocks per trajectory, each with a share of its
//         tokens: mark retired tokens, protect the pending prefix, pick the
//         fill tokens by an exact radix select on 64-bit keys (fill score,
//         token index; histograms summed over the cluster's shared memory),
//         and write I_j ascending;
// gather  16-byte vector copies of the retained K and V rows of every
//         (layer, KV head), plus positions; into caller buffers, or in place
//         (the retained rows move to rows 0..|I|-1 of the cache itself).
#include <cooperative_groups.h>
#include <type_traits>

#include "ckv_internal.cuh"

namespace ckv {
namespace {

constexpr int kThreads = 1024;
constexpr int kMaxPending = 2048;
// Blocks per trajectory (one cluster): one up to kOneBlock tokens, else eight.
// One block's dozen sweeps over 36.9K tokens took 62 us, most of it waiting
// for its own loads and for histogram additions to the same bin; eight take
// 33 us.  At 2,400 tokens one takes 11 us, eight 15; at 7,500 17 to 20 and
// 17 to 18, at 10,000 24 to 28 and 18 to 20.
constexpr int kCluster = 8;
constexpr int kOneBlock = 8192;
constexpr int kKeys = 8;   // tokens a thread keeps in registers; longer shares are read from memory every time

__device__ __forceinline__ uint64_t fill_key(float f, int i) {
  uint32_t u = __float_as_uint(f == 0.0f ? 0.0f : f);  // -0 and +0 tie
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);       // order-preserving
  return ((uint64_t)u << 32) | (uint32_t)i;              // ties: higher index first
}

// Block-wide exclusive scan of one int per thread; returns the total.
__device__ int block_scan(int v, int *excl, int *s_warp) {
  int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = lane < kThreads / 32 ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_warp[lane] = w;  // inclusive prefix of warp totals
  }
  __syncthreads();
  int before = warp ? s_warp[warp - 1] : 0;
  *excl = before + x - v;
  int total = s_warp[kThreads / 32 - 1];
  __syncthreads();
  return total;
}

// Adds one to a bin: the lanes that share the first active lane's bin (most
// scores of one magnitude do, in the top digit) add up first.
__device__ __forceinline__ void count_bin(unsigned *hist, bool active, unsigned bin) {
  const unsigned act = __ballot_sync(0xffffffffu, active);
  if (!act) return;
  const int lead = __ffs(act) - 1, lane = threadIdx.x % 32;
  const unsigned first = __shfl_sync(0xffffffffu, bin, lead);
  const unsigned same = __ballot_sync(0xffffffffu, active && bin == first);
  if (lane == lead) atomicAdd(&hist[first], (unsigned)__popc(same));
  else if (active && bin != first) atomicAdd(&hist[bin], 1u);
}

__global__ void __launch_bounds__(kThreads, 1) select_kernel(const __grid_constant__ CompactLaunch L, WsHeader *hdr) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int nb = cl.num_blocks(), t = blockIdx.x / nb, part = cl.block_rank();
  const TrajDev &tr = L.t[t];
  const int S = tr.S, P = tr.P;
  // this block's tokens
  const int share = (S + nb - 1) / nb, lo = min(S, part * share), hi = min(S, lo + share);
  // this thread's tokens, contiguous
  const int seg = (share + kThreads - 1) / kThreads;
  const int i0 = min(hi, lo + (int)threadIdx.x * seg), i1 = min(hi, i0 + seg);
  const bool in_regs = seg <= kKeys;
  uint8_t *cls = L.cls[t];  // 0 = fill candidate, 1 = retired, 2 = protected, 3 = kept
  __shared__ int s_warp[32];
  __shared__ int s_bad, s_prot_tokens, s_rem;
  __shared__ int s_pid[kMaxPending];
  __shared__ float s_pr[kMaxPending];
  __shared__ int2 s_span[kMaxPending];  // start and length of the live pending pages in their order
  __shared__ int s_live;
  __shared__ unsigned s_hist[2][256];  // this block's counts (alternate digits alternate buffers)
  __shared__ unsigned s_all[256];      // the cluster's counts
  __shared__ unsigned long long s_prefix;
  __shared__ int s_krem, s_exact;
  auto sync = [&]() {  // the cluster's barrier; a single block needs only its own
    if (nb > 1) cl.sync();
    else __syncthreads();
  };
  // sum over the cluster of an int in shared memory, after a barrier of the
  // cluster; `before` also gets the sum over the lower-ranked blocks
  auto total_of = [&](int *x, int *before) {
    sync();
    int sum = *x, low = 0;
    if (nb > 1) sum = 0;
    for (int r = 0; r < nb && nb > 1; ++r) {
      const int v = *cl.map_shared_rank(x, r);
      sum += v;
      if (r < part) low += v;
    }
    if (before) *before = low;
    return sum;
  };

  if (threadIdx.x == 0) {
    s_bad = 0;
    s_live = 0;
    s_rem = 0;
  }
  __syncthreads();
  for (int i = lo + threadIdx.x; i < hi; i += kThreads) {
    cls[i] = 0;
    if (isnan(L.fill[t][i])) s_bad = 1;
  }
  sync();
  // retired pages (D_c) are excluded
  for (int E = part * kThreads + threadIdx.x; E < P; E += nb * kThreads) {
    int ps = tr.ps[E], pl = tr.pl[E];
    if (pl < 0 || ps < 0 || ps > S - pl) {
      s_bad = 1;
      continue;
    }
    if (L.retired[t][E])
      for (int i = ps; i < ps + pl; ++i) cls[i] = 1;
  }
  // pending pages (every block orders them all): drop retired ones, order by (priority desc, page index asc)
  int np = L.n_pending[t];
  for (int k = threadIdx.x; k < np; k += kThreads) {
    int E = L.pending[t][k];
    float pr = (E >= 0 && E < P) ? L.prio[t][E] : 0.0f;
    if (E < 0 || E >= P || isnan(pr)) {
      s_bad = 1;
      E = -1;
    } else if (L.retired[t][E]) {
      E = -1;
    }
    s_pid[k] = E;
    s_pr[k] = pr;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < np; k += kThreads) {
    int E = s_pid[k];
    if (E < 0) continue;
    float pr = s_pr[k];
    int rank = 0;
    for (int j = 0; j < np; ++j) {
      int F = s_pid[j];
      if (F < 0) continue;
      if (F == E && j != k) s_bad = 1;  // duplicate page id
      rank += (s_pr[j] > pr) || (s_pr[j] == pr && F < E);
    }
    s_span[rank] = make_int2(tr.ps[E], tr.pl[E]);
    atomicAdd(&s_live, 1);
  }
  __syncthreads();
  const int bad = total_of(&s_bad, nullptr);
  // Every check above has run (NaN fill scores, page spans, pending ids,
  // duplicates): a failed one ends the trajectory here, before any page span
  // is used to index the class bytes or a duplicate leaves a rank unwritten.
  if (bad) {
    if (threadIdx.x == 0 && part == 0) {
      record_error(hdr, COMMITKV_ERR_DEVICE_INPUT, -5);
      L.n_idx[t] = 0;
    }
    sync();  // no block leaves while another reads its shared memory
    return;
  }
  if (threadIdx.x == 0) {
    // live entries occupy ranks [0, s_live); take the longest prefix that
    // fits both the page cap and the token budget B_N (Eq. 12)
    int pages = 0, toks = 0;
    for (; pages < s_live; ++pages) {
      const int len = s_span[pages].y;
      if (pages + 1 > L.cap || toks + len > L.B_N) break;
      toks += len;
    }
    s_prot_tokens = toks;
    s_live = pages;
  }
  __syncthreads();
  for (int k = threadIdx.x / 32; k < s_live; k += kThreads / 32) {  // a warp per page
    const int e = min(hi, s_span[k].x + s_span[k].y);
    for (int i = max(lo, s_span[k].x) + threadIdx.x % 32; i < e; i += 32) cls[i] = 2;
  }
  __syncthreads();
  // fill: other non-retired tokens by (score desc, index desc) within the room
  uint32_t key32[kKeys];   // in_regs: the upper halves of the thread's keys
  unsigned open = 0, kept = 0;  // in_regs, a bit per token: a fill candidate; protected or kept
  int rem_local = 0;
  if (in_regs) {
#pragma unroll
    for (int k = 0; k < kKeys; ++k) {
      key32[k] = 0;
      if (k < seg && i0 + k < i1) {
        const int c = cls[i0 + k];
        key32[k] = (uint32_t)(fill_key(L.fill[t][i0 + k], 0) >> 32);
        open |= (c == 0 ? 1u : 0u) << k;
        kept |= (c == 2 ? 1u : 0u) << k;
      }
    }
    rem_local = __popc(open);
  } else {
    for (int i = i0; i < i1; ++i) rem_local += cls[i] == 0;
  }
  if (threadIdx.x == 0) s_rem = 0;
  __syncthreads();
  rem_local = warp_sum_i(rem_local);
  if (threadIdx.x % 32 == 0) atomicAdd(&s_rem, rem_local);
  const int rem = total_of(&s_rem, nullptr);
  int room = L.B - s_prot_tokens;
  if (rem > room) {
    // exact k-th largest key (k = room) by 8-bit MSB-first radix select
    if (threadIdx.x == 0) {
      s_prefix = 0ull;
      s_krem = room;
      s_exact = 0;
    }
    unsigned long long mask = 0ull;
    // stops early once every key with the chosen prefix is taken: the
    // prefix (lower bits zero) is then itself the threshold
    for (int shift = 56; shift >= 0 && room > 0; shift -= 8) {
      // last read by the cluster two digits ago
      unsigned *hist = s_hist[(shift >> 3) & 1];
      if (threadIdx.x < 256) hist[threadIdx.x] = 0;
      __syncthreads();
      unsigned long long prefix = s_prefix;
      if (in_regs) {
#pragma unroll
        for (int k = 0; k < kKeys; ++k) {
          if (k >= seg) break;
          const uint64_t key = ((uint64_t)key32[k] << 32) | (uint32_t)(i0 + k);
          count_bin(hist, ((open >> k) & 1u) && (key & mask) == prefix, (unsigned)(key >> shift) & 255u);
        }
      } else {
        for (int k = 0; k < seg; ++k) {
          const int i = min(i0 + k, hi - 1);
          const bool mine = i0 + k < i1 && cls[i] == 0;
          const uint64_t key = mine ? fill_key(L.fill[t][i], i) : 0ull;
          count_bin(hist, mine && (key & mask) == prefix, (unsigned)(key >> shift) & 255u);
        }
      }
      sync();
      if (nb > 1) {
        if (threadIdx.x < 256) {  // every block sums the counts and finds the same bin
          unsigned sum = 0;
          for (int r = 0; r < nb; ++r) sum += cl.map_shared_rank(hist, r)[threadIdx.x];
          s_all[threadIdx.x] = sum;
        }
        __syncthreads();
        hist = s_all;
      }
      if (threadIdx.x < 32) {
        // the first bin, from the top, at which the count of larger keys
        // reaches `need`: lane l holds bins 255 - 8 l down to 248 - 8 l, a
        // warp scan gives each lane the count above its bins, and the lane
        // whose bins hold the crossing walks them in order
        const int lane = threadIdx.x, need = s_krem;
        unsigned sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) sum += hist[255 - 8 * lane - u];
        unsigned incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, incl >= (unsigned)need);
        if (hit != 0u && lane == __ffs(hit) - 1) {
          unsigned cum = incl - sum;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const unsigned c = hist[255 - 8 * lane - u];
            if (cum + c >= (unsigned)need) {
              s_prefix = prefix | ((unsigned long long)(255 - 8 * lane - u) << shift);
              s_krem = need - (int)cum;
              s_exact = s_krem == (int)c;
              break;
            }
            cum += c;
          }
        }
      }
      mask |= 255ull << shift;
      __syncthreads();
      if (s_exact) break;
    }
    const unsigned long long thr = s_prefix;
    if (in_regs) {
#pragma unroll
      for (int k = 0; k < kKeys; ++k)
        if (((open >> k) & 1u) && room > 0 && (((uint64_t)key32[k] << 32) | (uint32_t)(i0 + k)) >= thr) kept |= 1u << k;
    } else {
      for (int i = i0; i < i1; ++i)
        if (cls[i] == 0 && (room > 0 && fill_key(L.fill[t][i], i) >= thr)) cls[i] = 3;
    }
  } else if (in_regs) {
    kept |= open;
  } else {
    for (int i = i0; i < i1; ++i)
      if (cls[i] == 0) cls[i] = 3;
  }
  __syncthreads();
  // I_j ascending: protected (2) and kept (3) tokens of the threads' segments;
  // a block scan and the lower blocks' totals place them
  int cnt = __popc(kept);
  if (!in_regs) {
    cnt = 0;
    for (int i = i0; i < i1; ++i) cnt += cls[i] >= 2;
  }
  int excl, before;
  const int mine = block_scan(cnt, &excl, s_warp);
  if (threadIdx.x == 0) s_krem = mine;
  const int total = total_of(&s_krem, &before);
  for (int i = i0, o = before + excl; i < i1 && o < L.B; ++i)
    if (in_regs ? (kept >> (i - i0)) & 1u : cls[i] >= 2) L.idx[t][o++] = i;
  if (threadIdx.x == 0 && part == 0) L.n_idx[t] = total < L.B ? total : L.B;
  sync();  // no block leaves while another reads its shared memory
}

template <int VEC_BYTES>
__global__ void __launch_bounds__(256) gather_kernel(const __grid_constant__ CompactLaunch L) {
  int t = blockIdx.z;
  const TrajDev &tr = L.t[t];
  int slice = blockIdx.y;  // l * H + h
  int l = slice / L.H, h = slice % L.H;
  int row_bytes = L.d * L.elem_bytes;
  int vec_per_row = row_bytes / VEC_BYTES;
  int n = L.n_idx[t];
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int j = (int)(g / vec_per_row), vv = (int)(g % vec_per_row);
  if (j >= n) return;
  int i = L.idx[t][j];
  const char *ks = static_cast<const char *>(tr.k) + ((int64_t)l * tr.sl + (int64_t)h * tr.sh + (int64_t)i * tr.st) * L.elem_bytes;
  const char *vs = static_cast<const char *>(tr.v) + ((int64_t)l * tr.sl + (int64_t)h * tr.sh + (int64_t)i * tr.st) * L.elem_bytes;
  int64_t doff = (((int64_t)slice * L.B) + j) * row_bytes + (int64_t)vv * VEC_BYTES;
  if (L.k_out[t]) {
    if (VEC_BYTES == 16)
      *reinterpret_cast<uint4 *>(static_cast<char *>(L.k_out[t]) + doff) =
          *reinterpret_cast<const uint4 *>(ks + vv * VEC_BYTES);
    else
      *reinterpret_cast<uint16_t *>(static_cast<char *>(L.k_out[t]) + doff) =
          *reinterpret_cast<const uint16_t *>(ks + vv * VEC_BYTES);
  }
  if (L.v_out[t]) {
    if (VEC_BYTES == 16)
      *reinterpret_cast<uint4 *>(static_cast<char *>(L.v_out[t]) + doff) =
          *reinterpret_cast<const uint4 *>(vs + vv * VEC_BYTES);
    else
      *reinterpret_cast<uint16_t *>(static_cast<char *>(L.v_out[t]) + doff) =
          *reinterpret_cast<const uint16_t *>(vs + vv * VEC_BYTES);
  }
  if (slice == 0 && vv == 0 && L.pos_out[t]) L.pos_out[t][j] = tr.pos[i];
}

// In-place gather: one block per (K or V, layer, KV head, trajectory)
// slice.  I is strictly increasing with I_j >= j, so row j's destination is
// a source only for rows k <= j.  The block walks the slice in chunks of
// ROWS rows: it reads every source row of the chunk, waits at the barrier,
// then writes the chunk's destinations.  A destination in chunk c is read,
// if at all, by a row of chunk c or earlier, before that chunk's barrier;
// sources of later chunks lie at or after their own rows, past every row
// written so far.  Rows with I_j = j are left alone.
template <int VEC_BYTES, int ROWS>
__global__ void __launch_bounds__(256) gather_in_place_kernel(const __grid_constant__ CompactLaunch L) {
  using Vec = typename std::conditional<VEC_BYTES == 16, uint4, uint16_t>::type;
  constexpr int kMaxVec = 512 / VEC_BYTES;  // vectors per row at most (fp32, d = 128)
  constexpr int kPer = ROWS * kMaxVec / 256;
  const int t = blockIdx.z, slice = blockIdx.y;
  const TrajDev &tr = L.t[t];
  const int l = slice / L.H, h = slice % L.H;
  const int vpr = L.d * L.elem_bytes / VEC_BYTES;
  char *base = static_cast<char *>(const_cast<void *>(blockIdx.x ? tr.v : tr.k)) +
               ((int64_t)l * tr.sl + (int64_t)h * tr.sh) * L.elem_bytes;
  const int64_t rs = tr.st * L.elem_bytes;
  const int n = L.n_idx[t];
  const int32_t *idx = L.idx[t];
  for (int j0 = 0; j0 < n; j0 += ROWS) {
    Vec buf[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int e = threadIdx.x + 256 * u, r = e / vpr, w = e % vpr;
      if (r < ROWS && j0 + r < n) {
        const int i = idx[j0 + r];
        if (i != j0 + r) buf[u] = *reinterpret_cast<const Vec *>(base + i * rs + w * VEC_BYTES);
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int e = threadIdx.x + 256 * u, r = e / vpr, w = e % vpr;
      if (r < ROWS && j0 + r < n) {
        const int i = idx[j0 + r];
        if (i != j0 + r) *reinterpret_cast<Vec *>(base + (int64_t)(j0 + r) * rs + w * VEC_BYTES) = buf[u];
      }
    }
  }
}

// Positions in place, one block per trajectory, by the same chunk rule.
__global__ void __launch_bounds__(256) positions_in_place_kernel(const __grid_constant__ CompactLaunch L) {
  const int t = blockIdx.x;
  int32_t *pos = const_cast<int32_t *>(L.t[t].pos);
  const int n = L.n_idx[t];
  const int32_t *idx = L.idx[t];
  for (int j0 = 0; j0 < n; j0 += 256) {
    const int j = j0 + threadIdx.x;
    int v = 0;
    if (j < n) v = pos[idx[j]];
    __syncthreads();
    if (j < n) pos[j] = v;
  }
}

}  // namespace

cudaError_t launch_compact(const CompactLaunch &L, WsHeader *hdr, cudaStream_t stream) {
  if (L.n_traj <= 0) return cudaSuccess;
  int smax = 0;
  for (int t = 0; t < L.n_traj; ++t) smax = L.t[t].S > smax ? L.t[t].S : smax;
  const int nb = smax > kOneBlock ? kCluster : 1;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = nb;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L.n_traj * nb);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  ++launch_count();
  cudaError_t e = cudaLaunchKernelEx(&cfg, select_kernel, L, hdr);
  if (e != cudaSuccess) return e;
  if (L.in_place) {
    bool aligned = (L.d * L.elem_bytes) % 16 == 0;
    for (int t = 0; t < L.n_traj; ++t) {
      const TrajDev &tr = L.t[t];
      aligned &= ((uintptr_t)tr.k % 16 == 0) && ((uintptr_t)tr.v % 16 == 0) &&
                 ((tr.sl * L.elem_bytes) % 16 == 0) && ((tr.sh * L.elem_bytes) % 16 == 0) &&
                 ((tr.st * L.elem_bytes) % 16 == 0);
    }
    if (L.B == 0) return cudaSuccess;
    dim3 grid(2, L.M * L.H, L.n_traj);
    if (aligned) gather_in_place_kernel<16, 64><<<grid, 256, 0, stream>>>(L);
    else gather_in_place_kernel<2, 8><<<grid, 256, 0, stream>>>(L);
    launch_count() += 2;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    positions_in_place_kernel<<<L.n_traj, 256, 0, stream>>>(L);
    return cudaGetLastError();
  }
  bool any_out = false;
  bool aligned = (L.d * L.elem_bytes) % 16 == 0;
  for (int t = 0; t < L.n_traj; ++t) {
    any_out |= L.k_out[t] || L.v_out[t] || L.pos_out[t];
    const TrajDev &tr = L.t[t];
    aligned &= ((uintptr_t)tr.k % 16 == 0) && ((uintptr_t)tr.v % 16 == 0) &&
               ((tr.sl * L.elem_bytes) % 16 == 0) && ((tr.sh * L.elem_bytes) % 16 == 0) &&
               ((tr.st * L.elem_bytes) % 16 == 0) &&
               ((uintptr_t)L.k_out[t] % 16 == 0) && ((uintptr_t)L.v_out[t] % 16 == 0);
  }
  if (!any_out || L.B == 0) return cudaSuccess;
  int row_bytes = L.d * L.elem_bytes;
  if (aligned) {
    int64_t threads = (int64_t)L.B * (row_bytes / 16);
    dim3 grid((unsigned)((threads + 255) / 256), L.M * L.H, L.n_traj);
    gather_kernel<16><<<grid, 256, 0, stream>>>(L);
  } else {
    int64_t threads = (int64_t)L.B * (row_bytes / 2);
    dim3 grid((unsigned)((threads + 255) / 256), L.M * L.H, L.n_traj);
    gather_kernel<2><<<grid, 256, 0, stream>>>(L);
  }
  ++launch_count();
  return cudaGetLastError();
}

int compact_max_pending() { return kMaxPending; }

}  // namespace ckv
