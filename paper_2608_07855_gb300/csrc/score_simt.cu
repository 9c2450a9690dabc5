// Page deletion effects (Section 3.2, Eq. 6-8) — portable CUDA-core path.
//
// Three launches per call:
//   pass A   per (trajectory, layer, KV head, token chunk, row block):
//            online-softmax partials (max, sum, sum e*v, visible count) of
//            every probe row over the chunk;
//   combine  per probe row: merge the chunk partials into the row's final
//            max m, sum l, visible count n and output o (the stats);
//   pass B   per (trajectory, layer, KV head, page group, row block):
//            for each page E, S_E = sum_{i in E visible} e_i and
//            U_E = sum e_i v_i with e_i = exp(s_i - m), then
//            r = ||U_E - S_E o|| / ((l - S_E) ||o||)  (Eq. 6 with a = e / l),
//            max over the block's rows into R[E] and R_head[l][h][E] (Eq. 7).
// Scores are kept in base-2 units (scale * log2 e), fp32 throughout.
//
// A warp takes eight probe rows together: a lane holds two tokens of the
// 64-token tile (K read once for the eight rows, four channels at a time) and,
// for P V, D / 32 channels.  Row by row, with scalar loads, the fp32 Tiny
// workload (2K tokens, one layer, two heads) spent 161 us in pass A and 179 us
// in pass B, now 18 and 24; it is bound by latency, so small calls also take
// shorter chunks and fewer pages per block (see api.cu).  Four layers, four
// heads of 128 channels, 5K tokens: 1,190 -> 619 and 1,739 -> 619 us.
#include "ckv_internal.cuh"
#include "sm103.cuh"

namespace ckv {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRB = 64;               // probe rows per block
constexpr int kRowsPerWarp = kRB / kWarps;
constexpr int kTK = 64;               // tokens per shared-memory tile
constexpr float kNegInf = -__builtin_huge_valf();

__device__ __forceinline__ int find_traj(const int32_t *off, int n, int unit) {
  int t = 0;
  while (t + 1 < n && unit >= off[t + 1]) ++t;
  return t;
}

template <typename T, int D>
__device__ __forceinline__ void load_rows_q(const Batch &b, const TrajDev &tr, int l, int kvh,
                                            int row0, int rows, float *sQ) {
  const T *q = static_cast<const T *>(tr.q);
  for (int e = threadIdx.x; e < kRB * D; e += kThreads) {
    int r = e / D, c = e % D;
    float v = 0.0f;
    int row = row0 + r;
    if (row < rows) {
      int h = kvh * b.g + row / tr.W, w = row % tr.W;
      v = to_f32(q[(((int64_t)l * b.Hq + h) * tr.W + w) * D + c]);
    }
    sQ[r * D + c] = v;
  }
}

template <typename T, int D>
__device__ __forceinline__ void load_tile_kv(const TrajDev &tr, int l, int kvh, int tok0, int nt,
                                             float *sK, float *sV, int *sPos) {
  const T *kp = static_cast<const T *>(tr.k) + (int64_t)l * tr.sl + (int64_t)kvh * tr.sh;
  const T *vp = static_cast<const T *>(tr.v) + (int64_t)l * tr.sl + (int64_t)kvh * tr.sh;
  for (int e = threadIdx.x; e < kTK * D; e += kThreads) {
    int i = e / D, c = e % D;
    float kv = 0.0f, vv = 0.0f;
    if (i < nt) {
      int64_t off = (int64_t)(tok0 + i) * tr.st + c;
      kv = to_f32(kp[off]);
      vv = to_f32(vp[off]);
    }
    sK[i * (D + 4) + c] = kv;
    sV[i * D + c] = vv;
  }
  for (int i = threadIdx.x; i < kTK; i += kThreads) sPos[i] = i < nt ? tr.pos[tok0 + i] : 0x7fffffff;
}

// Scaled dot products of the warp's rows with tokens lane and lane + 32 of the
// tile (base 2).  bf16: every score one chain over the channels.  Statistics that a caller
// gives are mostly sums in that order, and the effects are differences in which
// it cancels: 12 to 16 layers of 64 channels, errors of 1.2e-6 to 5.3e-6
// against 2.9e-6 to 2.0e-5 with two chains.  fp32: two chains (even and odd
// channels) in packed FMAs, the smaller errors there (effects 3e-7 against
// 5e-7) and less latency (2K tokens: pass B 24 us against 32).
template <typename T, int D>
__device__ __forceinline__ void tile_scores(const float *q, const float *sK, int lane, float scale_log2,
                                            float (&s)[kRowsPerWarp][2]) {
  if constexpr (sizeof(T) == 2) {
    float a0[kRowsPerWarp], a1[kRowsPerWarp];
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) a0[k] = a1[k] = 0.0f;
#pragma unroll 2
    for (int c = 0; c < D; c += 4) {
      const float4 x = *reinterpret_cast<const float4 *>(sK + lane * (D + 4) + c);
      const float4 y = *reinterpret_cast<const float4 *>(sK + (lane + 32) * (D + 4) + c);
#pragma unroll
      for (int k = 0; k < kRowsPerWarp; ++k) {
        const float4 w = *reinterpret_cast<const float4 *>(q + k * D + c);
        a0[k] = fmaf(w.w, x.w, fmaf(w.z, x.z, fmaf(w.y, x.y, fmaf(w.x, x.x, a0[k]))));
        a1[k] = fmaf(w.w, y.w, fmaf(w.z, y.z, fmaf(w.y, y.y, fmaf(w.x, y.x, a1[k]))));
      }
    }
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) {
      s[k][0] = a0[k] * scale_log2;
      s[k][1] = a1[k] * scale_log2;
    }
  } else {
    using sm103::ffma2;
    float2 a0[kRowsPerWarp], a1[kRowsPerWarp];
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) a0[k] = a1[k] = make_float2(0.0f, 0.0f);
#pragma unroll 2
    for (int c = 0; c < D; c += 4) {
      const float4 x = *reinterpret_cast<const float4 *>(sK + lane * (D + 4) + c);
      const float4 y = *reinterpret_cast<const float4 *>(sK + (lane + 32) * (D + 4) + c);
#pragma unroll
      for (int k = 0; k < kRowsPerWarp; ++k) {
        const float4 w = *reinterpret_cast<const float4 *>(q + k * D + c);
        a0[k] = ffma2(make_float2(w.x, w.y), make_float2(x.x, x.y), a0[k]);
        a0[k] = ffma2(make_float2(w.z, w.w), make_float2(x.z, x.w), a0[k]);
        a1[k] = ffma2(make_float2(w.x, w.y), make_float2(y.x, y.y), a1[k]);
        a1[k] = ffma2(make_float2(w.z, w.w), make_float2(y.z, y.w), a1[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) {
      s[k][0] = (a0[k].x + a0[k].y) * scale_log2;
      s[k][1] = (a1[k].x + a1[k].y) * scale_log2;
    }
  }
}

// The lane's channels of row i of sV: lane, lane + 32, ...
template <int D>
__device__ __forceinline__ void v_row(const float *sV, int i, int lane, float (&v)[D / 32]) {
#pragma unroll
  for (int j = 0; j < D / 32; ++j) v[j] = sV[i * D + lane + 32 * j];
}

// The eight rows' weights of token i ([token][row] per warp).
__device__ __forceinline__ void p_rows(const float *pw, int i, float (&p)[kRowsPerWarp]) {
  static_assert(kRowsPerWarp == 8, "two float4 per token");
  const float4 a = *reinterpret_cast<const float4 *>(pw + i * kRowsPerWarp);
  const float4 b = *reinterpret_cast<const float4 *>(pw + i * kRowsPerWarp + 4);
  p[0] = a.x, p[1] = a.y, p[2] = a.z, p[3] = a.w, p[4] = b.x, p[5] = b.y, p[6] = b.z, p[7] = b.w;
}

// ---------------------------------------------------------------- pass A
template <typename T, int D>
__global__ void __launch_bounds__(kThreads) pass_a_kernel(const __grid_constant__ ScoreLaunch L,
                                                          float *partials) {
  extern __shared__ float smem[];
  float *sQ = smem;                       // [kRB][D]
  float *sK = sQ + kRB * D;               // [kTK][D + 4]
  float *sV = sK + kTK * (D + 4);         // [kTK][D]
  int *sPos = reinterpret_cast<int *>(sV + kTK * D);
  float *sP = reinterpret_cast<float *>(sPos + kTK);  // [kWarps][kTK][kRowsPerWarp]

  const Batch &b = L.batch;
  int unit = blockIdx.x;
  int t = find_traj(L.unit_off_a, b.n_traj, unit);
  const TrajDev &tr = b.t[t];
  int local = unit - L.unit_off_a[t];
  int nrb = L.nrb[t], nch = L.nchunk[t];
  int rb = local % nrb;
  local /= nrb;
  int c = local % nch;
  local /= nch;
  int kvh = local % b.H, li = local / b.H;
  int l = b.layer_ids[li];
  int rows = b.g * tr.W;
  int row0 = rb * kRB;
  int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  load_rows_q<T, D>(b, tr, l, kvh, row0, rows, sQ);

  constexpr int J = D / 32;
  float m_run[kRowsPerWarp], l_run[kRowsPerWarp], O[kRowsPerWarp][J];
  int n_run[kRowsPerWarp], qp[kRowsPerWarp];
#pragma unroll
  for (int k = 0; k < kRowsPerWarp; ++k) {
    m_run[k] = kNegInf;
    l_run[k] = 0.0f;
    n_run[k] = 0;
    int row = row0 + warp * kRowsPerWarp + k;
    qp[k] = row < rows ? tr.qpos[row % tr.W] : -0x7fffffff;
#pragma unroll
    for (int j = 0; j < J; ++j) O[k][j] = 0.0f;
  }

  int tok_begin = c * L.chunk_len;
  int tok_end = min(tr.S, tok_begin + L.chunk_len);
  for (int tok0 = tok_begin; tok0 < tok_end; tok0 += kTK) {
    int nt = min(kTK, tok_end - tok0);
    __syncthreads();
    load_tile_kv<T, D>(tr, l, kvh, tok0, nt, sK, sV, sPos);
    __syncthreads();
    float s[kRowsPerWarp][2];
    tile_scores<T, D>(sQ + warp * kRowsPerWarp * D, sK, lane, b.scale_log2, s);
    float *pw = sP + warp * kTK * kRowsPerWarp;
    unsigned live = 0;  // rows that see a token of this tile
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) {
      bool v0 = lane < nt && sPos[lane] <= qp[k], v1 = lane + 32 < nt && sPos[lane + 32] <= qp[k];
      const float mt = warp_max(fmaxf(v0 ? s[k][0] : kNegInf, v1 ? s[k][1] : kNegInf));
      const float m_new = fmaxf(m_run[k], mt);
      live |= (mt != kNegInf ? 1u : 0u) << k;
      // nothing visible in this tile: every weight is 0 and the sums stay
      const float alpha = m_run[k] == m_new ? 1.0f : exp2f(m_run[k] - m_new);
      const float p0 = v0 ? exp2f(s[k][0] - m_new) : 0.0f;
      const float p1 = v1 ? exp2f(s[k][1] - m_new) : 0.0f;
      l_run[k] = l_run[k] * alpha + warp_sum(p0 + p1);
      n_run[k] += __popc(__ballot_sync(0xffffffffu, v0)) + __popc(__ballot_sync(0xffffffffu, v1));
      m_run[k] = m_new;
      pw[lane * kRowsPerWarp + k] = p0;
      pw[(lane + 32) * kRowsPerWarp + k] = p1;
#pragma unroll
      for (int j = 0; j < J; ++j) O[k][j] *= alpha;
    }
    __syncwarp();
    if (live == (1u << kRowsPerWarp) - 1u) {
#pragma unroll 2
      for (int i = 0; i < nt; ++i) {
        float p[kRowsPerWarp], v[J];
        p_rows(pw, i, p);
        v_row<D>(sV, i, lane, v);
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k)
#pragma unroll
          for (int j = 0; j < J; ++j) O[k][j] = fmaf(p[k], v[j], O[k][j]);
      }
    } else if (live) {  // a row that sees nothing here is not touched (0 times an infinite value)
      for (int i = 0; i < nt; ++i) {
        float p[kRowsPerWarp], v[J];
        p_rows(pw, i, p);
        v_row<D>(sV, i, lane, v);
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k)
          if ((live >> k) & 1u) {
#pragma unroll
            for (int j = 0; j < J; ++j) O[k][j] = fmaf(p[k], v[j], O[k][j]);
          }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int k = 0; k < kRowsPerWarp; ++k) {
    int r = warp * kRowsPerWarp + k;
    float *dst = partials + ((int64_t)unit * kRB + r) * (D + 4);
    if (lane == 0) {
      dst[0] = m_run[k];
      dst[1] = l_run[k];
      dst[2] = (float)n_run[k];
      dst[3] = 0.0f;
    }
#pragma unroll
    for (int j = 0; j < J; ++j) dst[4 + lane + 32 * j] = O[k][j];
  }
}

// ---------------------------------------------------------------- combine
// One warp per probe row of the selected layers.
template <int D>
__global__ void __launch_bounds__(kThreads) combine_kernel(const __grid_constant__ ScoreLaunch L,
                                                           const float *partials) {
  const Batch &b = L.batch;
  int gw = (blockIdx.x * kThreads + threadIdx.x) / 32, lane = threadIdx.x % 32;
  int total = L.row_off[b.n_traj];
  if (gw >= total) return;
  int t = find_traj(L.row_off, b.n_traj, gw);
  const TrajDev &tr = b.t[t];
  int local = gw - L.row_off[t];
  int rows = b.g * tr.W;
  int row = local % rows;  // row within (layer, KV head)
  local /= rows;
  int kvh = local % b.H, li = local / b.H;
  int l = b.layer_ids[li];
  int nrb = L.nrb[t], nch = L.nchunk[t];
  int rb = row / kRB, rl = row % kRB;
  auto part = [&](int c) {
    int unit = L.unit_off_a[t] + (((li * b.H + kvh) * nch + c) * nrb + rb);
    return partials + ((int64_t)unit * kRB + rl) * (D + 4);
  };
  float m = kNegInf;
  for (int c = lane; c < nch; c += 32) m = fmaxf(m, part(c)[0]);
  m = warp_max(m);
  constexpr int J = D / 32;
  float o[J];
#pragma unroll
  for (int j = 0; j < J; ++j) o[j] = 0.0f;
  float lsum = 0.0f, n = 0.0f;
#pragma unroll 4
  for (int c = 0; c < nch; ++c) {
    const float *p = part(c);
    const float pm = p[0];
    float v[J];
#pragma unroll
    for (int j = 0; j < J; ++j) v[j] = p[4 + lane + 32 * j];
    n += p[2];
    const float a = pm == kNegInf ? 0.0f : exp2f(pm - m);
    lsum = fmaf(p[1], a, lsum);
#pragma unroll
    for (int j = 0; j < J; ++j) o[j] = fmaf(pm == kNegInf ? 0.0f : v[j], a, o[j]);
  }
  float inv = lsum > 0.0f ? 1.0f / lsum : 0.0f;
  int h = kvh * b.g + row / tr.W, w = row % tr.W;
  float *dst = L.stats[t] + (((int64_t)l * b.Hq + h) * tr.W + w) * (D + 4);
  if (lane == 0) {
    dst[0] = m == kNegInf ? m : m / 1.4426950408889634f;  // natural units
    dst[1] = lsum;
    dst[2] = n;
    dst[3] = 0.0f;
  }
#pragma unroll
  for (int j = 0; j < J; ++j) dst[4 + lane + 32 * j] = o[j] * inv;
}

// ---------------------------------------------------------------- pass B
constexpr int kPG = 16;  // pages per block at most

// x[k] on lane 4 k .. 4 k + 3.
template <typename X>
__device__ __forceinline__ X of_lane(const X (&x)[kRowsPerWarp], int lane) {
  // halving selects (a chain of equal compares becomes an indexed access to
  // local memory)
  X r[kRowsPerWarp];
#pragma unroll
  for (int k = 0; k < kRowsPerWarp; ++k) r[k] = x[k];
#pragma unroll
  for (int n = kRowsPerWarp / 2, bit = 16; n > 0; n /= 2, bit /= 2)
#pragma unroll
    for (int k = 0; k < n; ++k) r[k] = (lane & bit) ? r[k + n] : r[k];
  return r[0];
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads) pass_b_kernel(const __grid_constant__ ScoreLaunch L,
                                                          WsHeader *hdr) {
  extern __shared__ float smem[];
  float *sQ = smem;
  float *sK = sQ + kRB * D;
  float *sV = sK + kTK * (D + 4);
  int *sPos = reinterpret_cast<int *>(sV + kTK * D);
  float *sP = reinterpret_cast<float *>(sPos + kTK);
  float *sR = sP + kWarps * kTK * kRowsPerWarp;  // [kPG] block max per page

  const Batch &b = L.batch;
  int unit = blockIdx.x;
  int t = find_traj(L.unit_off_b, b.n_traj, unit);
  const TrajDev &tr = b.t[t];
  int local = unit - L.unit_off_b[t];
  int nrb = L.nrb[t], npg = L.npg[t];
  int rb = local % nrb;
  local /= nrb;
  int pg = local % npg;
  local /= npg;
  int kvh = local % b.H, li = local / b.H;
  int l = b.layer_ids[li];
  int rows = b.g * tr.W;
  int row0 = rb * kRB;
  int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  constexpr int J = D / 32;

  load_rows_q<T, D>(b, tr, l, kvh, row0, rows, sQ);
  // this warp's rows: final stats
  float m2[kRowsPerWarp], lsum[kRowsPerWarp], onorm[kRowsPerWarp], o[kRowsPerWarp][J];
  int nvis[kRowsPerWarp], qp[kRowsPerWarp], hrow[kRowsPerWarp];
#pragma unroll
  for (int k = 0; k < kRowsPerWarp; ++k) {
    int row = row0 + warp * kRowsPerWarp + k;
    bool ok = row < rows;
    int h = kvh * b.g + (ok ? row / tr.W : 0), w = ok ? row % tr.W : 0;
    hrow[k] = ok ? h : -1;
    const float *st = L.stats[t] + (((int64_t)l * b.Hq + h) * tr.W + w) * (D + 4);
    float mn = ok ? st[0] : kNegInf;
    m2[k] = mn == kNegInf ? mn : mn * 1.4426950408889634f;
    lsum[k] = ok ? st[1] : 0.0f;
    nvis[k] = ok ? L.nvis_w[t][w] : 0;
    qp[k] = ok ? tr.qpos[w] : -0x7fffffff;
    float ss = 0.0f;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      o[k][j] = ok ? st[4 + lane + 32 * j] : 0.0f;
      ss = fmaf(o[k][j], o[k][j], ss);
    }
    onorm[k] = sqrtf(warp_sum(ss));
  }

  // What Eq. 6 takes of row lane / 4: the lanes evaluate the warp's rows side
  // by side (every lane all eight, one after another, with a butterfly each,
  // was half of a page's time: 2K tokens of 64 fp32 channels 42 us, 24 so;
  // 5K tokens of 128 fp32 channels 773 us, 618 so).
  static_assert(kRowsPerWarp == 8, "four lanes per row");
  const float my_l = of_lane(lsum, lane), my_on = of_lane(onorm, lane);
  const int my_nvis = of_lane(nvis, lane), my_h = of_lane(hrow, lane);

  int E0 = pg * L.pages_per_block, E1 = min(tr.P, E0 + L.pages_per_block);
  for (int e = threadIdx.x; e < kPG; e += kThreads) sR[e] = 0.0f;
  __syncthreads();
  float *pw = sP + warp * kTK * kRowsPerWarp;
  float S_E[kRowsPerWarp], U[kRowsPerWarp][J];
  int n_E;  // of row lane / 4
  int w0 = 0, w1 = 0;  // tokens of the tile in shared memory
  unsigned seen0 = 0u, seen1 = 0u;  // the tile's visible tokens, row lane / 4
  for (int E = E0; E < E1; ++E) {
    int ps = tr.ps[E], pl = tr.pl[E];
    bool bad = pl < 0 || ps < 0 || ps > tr.S - pl || (E > 0 && ps < tr.ps[E - 1] + tr.pl[E - 1]);
    if (bad) {
      if (threadIdx.x == 0) record_error(hdr, COMMITKV_ERR_DEVICE_INPUT, E);
      continue;
    }
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) {
      S_E[k] = 0.0f;
#pragma unroll
      for (int j = 0; j < J; ++j) U[k][j] = 0.0f;
    }
    n_E = 0;
    for (int tok = ps; tok < ps + pl;) {
      if (tok < w0 || tok >= w1) {  // the next 64 tokens from here: several pages where they are short
        w0 = tok;
        w1 = min(tr.S, w0 + kTK);
        const int nt = w1 - w0;
        __syncthreads();
        load_tile_kv<T, D>(tr, l, kvh, w0, nt, sK, sV, sPos);
        __syncthreads();
        float s[kRowsPerWarp][2];
        unsigned seen[2][kRowsPerWarp];
        tile_scores<T, D>(sQ + warp * kRowsPerWarp * D, sK, lane, b.scale_log2, s);
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k) {
          const bool v0 = lane < nt && sPos[lane] <= qp[k], v1 = lane + 32 < nt && sPos[lane + 32] <= qp[k];
          pw[lane * kRowsPerWarp + k] = v0 ? exp2f(s[k][0] - m2[k]) : 0.0f;
          pw[(lane + 32) * kRowsPerWarp + k] = v1 ? exp2f(s[k][1] - m2[k]) : 0.0f;
          seen[0][k] = __ballot_sync(0xffffffffu, v0);
          seen[1][k] = __ballot_sync(0xffffffffu, v1);
        }
        seen0 = of_lane(seen[0], lane);
        seen1 = of_lane(seen[1], lane);
        __syncwarp();
      }
      const int i0 = tok - w0, i1 = min(ps + pl, w1) - w0;
      // the bits of tokens [i0, i1) of the tile
      auto bits = [&](int base) {
        const int a = max(i0 - base, 0), z = min(i1 - base, 32);
        return z <= a ? 0u : (z == 32 ? 0xffffffffu : (1u << z) - 1u) & ~((1u << a) - 1u);
      };
      n_E += __popc(seen0 & bits(0)) + __popc(seen1 & bits(32));
#pragma unroll 2
      for (int i = i0; i < i1; ++i) {
        float p[kRowsPerWarp], v[J];
        p_rows(pw, i, p);
        v_row<D>(sV, i, lane, v);
#pragma unroll
        for (int k = 0; k < kRowsPerWarp; ++k) {
          S_E[k] += p[k];
#pragma unroll
          for (int j = 0; j < J; ++j) U[k][j] = fmaf(p[k], v[j], U[k][j]);
        }
      }
      tok = w0 + i1;
    }
    float ss[kRowsPerWarp];
#pragma unroll
    for (int k = 0; k < kRowsPerWarp; ++k) {
      ss[k] = 0.0f;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        float dlt = fmaf(-S_E[k], o[k][j], U[k][j]);
        ss[k] = fmaf(dlt, dlt, ss[k]);
      }
    }
    // row lane / 4 on each lane: the butterfly's additions, each row's in an
    // eighth of the lanes from the third on
#pragma unroll
    for (int off = 16, n = kRowsPerWarp / 2; off > 0; off >>= 1, n /= 2) {
      if (n > 0) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
          const float keep = up ? ss[k + n] : ss[k], send = up ? ss[k] : ss[k + n];
          ss[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      } else {
        ss[0] += __shfl_xor_sync(0xffffffffu, ss[0], off);
      }
    }
    float r = 0.0f;
    if (my_h >= 0) {
      r = effect_value(n_E, my_nvis, of_lane(S_E, lane), my_l, ss[0], my_on);
      if (lane % 4 == 0 && L.headR[t]) atomic_max_nonneg(L.headR[t] + ((int64_t)l * b.Hq + my_h) * tr.P + E, r);
    }
    const unsigned rmax = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(0.0f, r)));
    if (lane == 0) atomicMax(reinterpret_cast<int *>(sR + (E - E0)), (int)rmax);
  }
  __syncthreads();
  for (int E = E0 + threadIdx.x; E < E1; E += kThreads) atomic_max_nonneg(L.R[t] + E, sR[E - E0]);
}

// Per trajectory and window position w: the number of resident tokens with
// pos <= qpos[w] (positions increase, so a binary search).  Also clears R, for
// the atomic maxima that follow.
__global__ void __launch_bounds__(256) count_visible_kernel(const __grid_constant__ ScoreLaunch L) {
  const int t = blockIdx.x;
  const TrajDev &tr = L.batch.t[t];
  for (int E = threadIdx.x; E < tr.P; E += blockDim.x) L.R[t][E] = 0.0f;
  for (int w = threadIdx.x; w < tr.W; w += blockDim.x) {
    const int qp = tr.qpos[w];
    int a = 0, b = tr.S;
    while (a < b) {
      int mid = (a + b) >> 1;
      if (tr.pos[mid] <= qp) a = mid + 1;
      else b = mid;
    }
    L.nvis_w[t][w] = a;
  }
}

template <typename T, int D>
cudaError_t launch_typed(const ScoreLaunch &L, float *partials, WsHeader *hdr, cudaStream_t s) {
  size_t smem = (size_t)(kRB * D + kTK * (D + 4) + kTK * D) * 4 + kTK * 4 + kWarps * kTK * kRowsPerWarp * 4 + kPG * 4;
  cudaError_t e;
  e = cudaFuncSetAttribute(pass_a_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(pass_b_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  count_visible_kernel<<<L.batch.n_traj, 256, 0, s>>>(L);
  int na = L.from_stats ? 0 : L.unit_off_a[L.batch.n_traj];
  if (na > 0) pass_a_kernel<T, D><<<na, kThreads, smem, s>>>(L, partials);
  int rows = L.from_stats ? 0 : L.row_off[L.batch.n_traj];
  if (rows > 0) combine_kernel<D><<<(rows * 32 + kThreads - 1) / kThreads, kThreads, 0, s>>>(L, partials);
  int nb = L.unit_off_b[L.batch.n_traj];
  if (nb > 0) pass_b_kernel<T, D><<<nb, kThreads, smem, s>>>(L, hdr);
  launch_count() += 1 + (na > 0) + (rows > 0) + (nb > 0);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_score_simt(const ScoreLaunch &L, float *partials, WsHeader *hdr,
                              cudaStream_t stream) {
  bool bf = L.batch.dtype == COMMITKV_BF16;
  if (L.batch.d == 128)
    return bf ? launch_typed<__nv_bfloat16, 128>(L, partials, hdr, stream)
              : launch_typed<float, 128>(L, partials, hdr, stream);
  return bf ? launch_typed<__nv_bfloat16, 64>(L, partials, hdr, stream)
            : launch_typed<float, 64>(L, partials, hdr, stream);
}

int simt_rows_per_block() { return kRB; }
int simt_pages_per_block() { return kPG; }

}  // namespace ckv
