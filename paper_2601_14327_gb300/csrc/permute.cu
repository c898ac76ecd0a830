// Dispatch and combine: the data movement around the grouped expert FFN.
//
// moe_permute is a stable counting sort of the T*k assignments by expert
// (order inside a group: token, then slot), so the grouped layout is
// deterministic and bit-exact. Groups start at multiples of 128 rows so that
// every 128-row GEMM tile belongs to one expert; padding rows are zero.
#include <cuda.h>
#include <limits.h>

#include <mutex>

#include "common.cuh"

MOE_DEV_ERR_DECL

namespace {

constexpr int kChunk = moe::kPermChunk;  // assignments per block
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kRankThreads = 1024;
constexpr int kRankWarps = kRankThreads / 32;
constexpr int kRankSteps = kChunk / kRankThreads;  // 32-wide steps of a warp
constexpr int kRankGroups = kRankThreads / 256;    // threads per expert in the prefix

// Block histograms: hist[b * E + e] = #{a in chunk b : idx[a] == e}.
__global__ void __launch_bounds__(kRankThreads) perm_hist_kernel(const int32_t *__restrict__ idx,
                                                                 int64_t A, int E,
                                                                 int32_t *__restrict__ hist) {
  __shared__ int sh[256];
  for (int e = threadIdx.x; e < E; e += blockDim.x) sh[e] = 0;
  __syncthreads();
  pdl_start();
  const int64_t a0 = int64_t(blockIdx.x) * kChunk;
  const int64_t a1 = min(A, a0 + kChunk);
  for (int64_t a = a0 + threadIdx.x; a < a1; a += blockDim.x) {
    const int e = idx[a];
    if (e >= 0 && e < E) atomicAdd(&sh[e], 1);
    else dev_flag(&g_dev_err, MOE_DEV_BAD_EXPERT);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += blockDim.x) hist[size_t(blockIdx.x) * E + e] = sh[e];
}

// Many chunks: the block histograms are summed over the chunks once, in place (afterwards
// hist[b * E + e] counts chunks 0..b), so that a rank block reads two of their rows and not all
// nblk: that pass is quadratic in the chunks. A block takes 32 experts, one per lane; its warps
// take kPrefixRows consecutive chunks each, kRankWarps * kPrefixRows per turn.
constexpr int kPrefixRows = 16;
__global__ void __launch_bounds__(kRankThreads) perm_prefix_kernel(int32_t *__restrict__ hist, int E, int nblk) {
  __shared__ int sum[kRankWarps][32];
  pdl_start();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
  int before = 0;  // of this expert in the chunks of earlier turns
  for (int b0 = 0; b0 < nblk; b0 += kRankWarps * kPrefixRows) {
    const int b1 = b0 + warp * kPrefixRows;
    int v[kPrefixRows];
#pragma unroll
    for (int i = 0; i < kPrefixRows; ++i) v[i] = e < E && b1 + i < nblk ? hist[size_t(b1 + i) * E + e] : 0;
#pragma unroll
    for (int i = 1; i < kPrefixRows; ++i) v[i] += v[i - 1];
    sum[warp][lane] = v[kPrefixRows - 1];
    __syncthreads();
    int own = before;
#pragma unroll 8
    for (int w = 0; w < kRankWarps; ++w) {
      const int c = sum[w][lane];
      if (w < warp) own += c;
      before += c;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPrefixRows; ++i)
      if (e < E && b1 + i < nblk) hist[size_t(b1 + i) * E + e] = own + v[i];
  }
}

// Row of every assignment: group start + rank among the earlier assignments of the same
// expert; group counts and padded group offsets (written by block 0). Latency-bound (a few
// 16 KB chunks), so a block does in registers and shared memory what took three launches:
// - ranks inside the block: warps own consecutive 128-assignment sub-chunks in 32-wide steps;
//   lanes with equal experts are ranked by lane order, earlier steps by a per-warp count;
// - the counts of the chunks before it and of all chunks, from the block histograms (one pass
//   over nblk * E entries from L2 per block, or their sums over the chunks from
//   perm_prefix_kernel; a single chunk needs no histogram kernel);
// - the scan of the padded group sizes (every block, 8 warps).
// Histogram + scan + rank kernels took 5.7 + 4.5 + 8.4 us and two gaps at T=16384, top-8, 64
// experts (32 chunks), 2.9 + 2.8 + 7.7 us at T=512, top-2; one kernel takes 5.2 us there now.
// MANY: hist holds the sums over the chunks, and 32 registers leave room for two blocks per SM
// (51 without that bound, which the few blocks of a small layout are faster with).
template <bool MANY>
__global__ void __launch_bounds__(kRankThreads, MANY ? 2 : 1) perm_rank_kernel(
    const int32_t *__restrict__ idx, int64_t A, int E, int nblk, const int32_t *__restrict__ hist,
    const int32_t *__restrict__ counts_check, int64_t rows_cap, int32_t *__restrict__ group_offsets,
    int32_t *__restrict__ group_counts, int32_t *__restrict__ row_of_assignment, int k,
    int32_t *__restrict__ token_of_row) {
  __shared__ int wh[kRankWarps][256];  // assignments of each warp to each expert, then their first row
  __shared__ int part[kRankGroups][2][256];
  __shared__ int s_warp[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = lane; i < E; i += 32) wh[warp][i] = 0;  // (only this warp uses it at first)
  __syncwarp();
  pdl_start();
  const int64_t a0 = int64_t(blockIdx.x) * kChunk + int64_t(warp) * (kRankSteps * 32) + lane;
  int e[kRankSteps], pos[kRankSteps];
#pragma unroll
  for (int s = 0; s < kRankSteps; ++s) {
    const int64_t a = a0 + s * 32;
    e[s] = -1;
    if (a < A) {
      e[s] = idx[a];
      if (e[s] < 0 || e[s] >= E) {
        e[s] = -1;
        dev_flag(&g_dev_err, MOE_DEV_BAD_EXPERT);
      }
    }
  }
  const int ex = tid & 255, grp = tid >> 8;
  if (nblk > 1) {
    int before = 0, all = 0;
    if (MANY) {
      if (grp == 0 && ex < E) {
        all = hist[size_t(nblk - 1) * E + ex];
        before = blockIdx.x > 0 ? hist[size_t(blockIdx.x - 1) * E + ex] : 0;
      }
    } else if (ex < E) {
#pragma unroll 8
      for (int b = grp; b < nblk; b += kRankGroups) {
        const int v = hist[size_t(b) * E + ex];
        all += v;
        if (b < int(blockIdx.x)) before += v;
      }
    }
    part[grp][0][ex] = before;
    part[grp][1][ex] = all;
  }
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int s = 0; s < kRankSteps; ++s) {
    const unsigned peers = __match_any_sync(0xffffffffu, e[s]);
    pos[s] = __popc(peers & lt);
    if (e[s] >= 0) pos[s] += wh[warp][e[s]];
    __syncwarp();
    if (e[s] >= 0 && lane == __ffs(peers) - 1) wh[warp][e[s]] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // thread ex of the first 256: the expert's counts per warp -> exclusive, its total, its group
  if (tid < 256) {
    int own = 0;
    if (ex < E) {
#pragma unroll 8
      for (int w = 0; w < kRankWarps; ++w) {
        const int c = wh[w][ex];
        wh[w][ex] = own;
        own += c;
      }
    }
    int before = 0, cnt = own;
    if (nblk > 1) {
      cnt = 0;
#pragma unroll
      for (int g = 0; g < kRankGroups; ++g) {
        before += part[g][0][ex];
        cnt += part[g][1][ex];
      }
    }
    if (ex >= E) cnt = 0;
    const int padded = (cnt + moe::kGroupPad - 1) / moe::kGroupPad * moe::kGroupPad;
    int incl = padded;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 31) s_warp[warp] = incl;
    asm volatile("bar.sync 1, 256;" ::: "memory");
    int base = incl - padded, total = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      if (w < warp) base += s_warp[w];
      total += s_warp[w];
    }
    const bool overflow = int64_t(total) > rows_cap;
    part[0][0][ex] = overflow ? INT_MIN : base + before;  // first row of this block's assignments
    if (blockIdx.x == 0) {
      if (ex < E) {
        group_offsets[ex] = base;
        group_counts[ex] = cnt;
        if (counts_check != nullptr && counts_check[ex] != cnt)
          dev_flag(&g_dev_err, MOE_DEV_COUNT_MISMATCH);
      }
      if (tid == 0) {
        group_offsets[E] = total;
        if (overflow) dev_flag(&g_dev_err, MOE_DEV_ROWS_OVERFLOW);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < kRankSteps; ++s) {
    const int64_t a = a0 + s * 32;
    if (a >= A) continue;
    int row = -1;
    if (e[s] >= 0 && part[0][0][e[s]] != INT_MIN) row = part[0][0][e[s]] + wh[warp][e[s]] + pos[s];
    row_of_assignment[a] = row;
    if (token_of_row != nullptr && row >= 0) token_of_row[row] = int(a / k);
  }
}

// Pad rows of every group read token 0 (their products are multiplied by zero
// downstream: the pad rows of d_out_perm and of the router's d_logits are zero).
__global__ void __launch_bounds__(kThreads) pad_token_kernel(const int32_t *__restrict__ group_offsets,
                                                             const int32_t *__restrict__ group_counts,
                                                             int E, int64_t rows_cap,
                                                             int32_t *__restrict__ token_of_row) {
  pdl_start();
  const int e = blockIdx.x;
  const int r0 = group_offsets[e] + group_counts[e];
  const int r1 = int(min((long long)group_offsets[e + 1], (long long)rows_cap));
  for (int r = r0 + threadIdx.x; r < r1; r += kThreads) token_of_row[r] = 0;
}

// Zeroes the padding rows [group_offsets[e] + group_counts[e], group_offsets[e+1]) of expert
// b / kPadSplit, share b % kPadSplit. The first E * kPadSplit blocks of the kernels that
// write a grouped tensor do this beside the token rows (as a launch of its own it took
// 8 us of a 240 us dispatch at T=16384, d=4096, 64 experts, and 2-3 us of a small one).
constexpr int kPadSplit = 8;
__device__ __forceinline__ void zero_pad_rows(int b, const int32_t *__restrict__ group_offsets,
                                              const int32_t *__restrict__ group_counts, int d,
                                              int64_t rows_cap, uint16_t *__restrict__ buf) {
  const int e = b / kPadSplit;
  const int r0 = group_offsets[e] + group_counts[e];
  const int r1 = int(min((long long)group_offsets[e + 1], (long long)rows_cap));
  const int nv = d / 8;
  const uint4 z = make_uint4(0, 0, 0, 0);
  for (int r = r0 + (b % kPadSplit) * kWarps + int(threadIdx.x >> 5); r < r1; r += kPadSplit * kWarps)
    for (int c = threadIdx.x & 31; c < nv; c += 32) stg_v4(buf + size_t(r) * d + c * 8, z);
}

// Token and column segment of a warp: nseg warps share a token, warp `seg` taking its 16-byte
// vectors lane + 32 (seg + nseg i) (see token_segments). False past the last token.
__device__ __forceinline__ bool token_segment(int block, int T, int nseg, int *t, int *seg) {
  const int w = block * kWarps + int(threadIdx.x >> 5);
  *t = w / nseg;
  *seg = w - *t * nseg;
  return *t < T;
}

// One warp (or nseg) per token: read x[t,:] once, write it to its k grouped rows. Blocks below
// pad_blocks zero padding rows.
// (SEG: nseg > 1; the fixed strides of the other form are worth 2% at T=16384.)
template <bool SEG>
__global__ void __launch_bounds__(kThreads) perm_gather_kernel(
    const uint16_t *__restrict__ x, const int32_t *__restrict__ row_of_assignment, int T, int d,
    int k, int nseg, int64_t rows_cap, int pad_blocks, const int32_t *__restrict__ group_offsets,
    const int32_t *__restrict__ group_counts, uint16_t *__restrict__ x_perm) {
  pdl_start();
  if (int(blockIdx.x) < pad_blocks) {
    zero_pad_rows(blockIdx.x, group_offsets, group_counts, d, rows_cap, x_perm);
    return;
  }
  const int lane = threadIdx.x & 31;
  int t, seg;
  if (!token_segment(blockIdx.x - pad_blocks, T, SEG ? nseg : 1, &t, &seg)) return;
  int my_row = (lane < k) ? row_of_assignment[size_t(t) * k + lane] : -1;
  int rows[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) rows[j] = __shfl_sync(0xffffffffu, my_row, j);
  const int nv = d / 8, step = SEG ? 32 * nseg : 32;
  const uint16_t *src = x + size_t(t) * d;
  // four 16-byte loads in flight per lane before their stores
  for (int c0 = lane + 32 * seg; c0 < nv; c0 += 4 * step) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + step * u < nv) v[u] = ldg_nc_v4(src + (c0 + step * u) * 8);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = c0 + step * u;
      if (c >= nv) break;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < k && rows[j] >= 0 && rows[j] < rows_cap) stg_v4(x_perm + size_t(rows[j]) * d + c * 8, v[u]);
    }
  }
}

// y[t] = sum_j g[t,j] * out_perm[row(t,j)]  (fp32 sum, one bf16 rounding)
__global__ void __launch_bounds__(kThreads) combine_kernel(
    const uint16_t *__restrict__ out_perm, const int32_t *__restrict__ row_of_assignment,
    const float *__restrict__ gate, int T, int d, int k, int nseg, uint16_t *__restrict__ y) {
  pdl_start();
  const int lane = threadIdx.x & 31;
  int t, seg;
  if (!token_segment(blockIdx.x, T, nseg, &t, &seg)) return;
  int my_row = (lane < k) ? row_of_assignment[size_t(t) * k + lane] : -1;
  float my_g = (lane < k) ? gate[size_t(t) * k + lane] : 0.f;
  int rows[8];
  float g[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    rows[j] = __shfl_sync(0xffffffffu, my_row, j);
    g[j] = __shfl_sync(0xffffffffu, my_g, j);
  }
  const int nv = d / 8;
  for (int c = lane + 32 * seg; c < nv; c += 32 * nseg) {
    uint4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < k && rows[j] >= 0) v[j] = ldg_nc_v4(out_perm + size_t(rows[j]) * d + c * 8);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < k && rows[j] >= 0) {
        float f[8];
        unpack8(v[j], f);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = fmaf(g[j], f[q], acc[q]);
      }
    }
    stg_v4(y + size_t(t) * d + c * 8, pack8(acc));
  }
}

// d_out_perm[row(t,j)] = g[t,j] * dy[t];  d_gate[t,j] = <dy[t], out_perm[row(t,j)]>
// DOUT: d_out_perm rows = g * dy[t]; DGATE: d_gate = <dy[t], out_perm rows>. The two
// halves can run as separate launches (DGATE alone reads out_perm and writes nothing
// large; DOUT alone never reads out_perm). Blocks below pad_blocks (DOUT only) zero
// padding rows of d_out_perm. nseg is 1 with DGATE, whose sums run over the whole row.
template <bool DOUT, bool DGATE>
__global__ void __launch_bounds__(kThreads) combine_bwd_kernel(
    const uint16_t *__restrict__ dy, const uint16_t *__restrict__ out_perm,
    const int32_t *__restrict__ row_of_assignment, const float *__restrict__ gate, int T, int d,
    int k, int nseg, int64_t rows_cap, int pad_blocks, const int32_t *__restrict__ group_offsets,
    const int32_t *__restrict__ group_counts, uint16_t *__restrict__ d_out_perm,
    float *__restrict__ d_gate) {
  pdl_start();
  if (DOUT && int(blockIdx.x) < pad_blocks) {
    zero_pad_rows(blockIdx.x, group_offsets, group_counts, d, rows_cap, d_out_perm);
    return;
  }
  const int lane = threadIdx.x & 31;
  int t, seg;
  if (!token_segment(blockIdx.x - pad_blocks, T, nseg, &t, &seg)) return;
  int my_row = (lane < k) ? row_of_assignment[size_t(t) * k + lane] : -1;
  float my_g = (lane < k) ? gate[size_t(t) * k + lane] : 0.f;
  int rows[8];
  float g[8], dot[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    rows[j] = __shfl_sync(0xffffffffu, my_row, j);
    if (rows[j] >= rows_cap) rows[j] = -1;
    g[j] = __shfl_sync(0xffffffffu, my_g, j);
    dot[j] = 0.f;
  }
  const int nv = d / 8;
  for (int c = lane + 32 * seg; c < nv; c += 32 * nseg) {
    float fd[8];
    unpack8(ldg_nc_v4(dy + size_t(t) * d + c * 8), fd);
    uint4 v[8];
    if (DGATE) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < k && rows[j] >= 0) v[j] = ldg_nc_v4(out_perm + size_t(rows[j]) * d + c * 8);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < k && rows[j] >= 0) {
        if (DGATE) {
          float f[8];
          unpack8(v[j], f);
#pragma unroll
          for (int q = 0; q < 8; ++q) dot[j] = fmaf(fd[q], f[q], dot[j]);
        }
        if (DOUT) {
          float o[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) o[q] = g[j] * fd[q];
          stg_v4(d_out_perm + size_t(rows[j]) * d + c * 8, pack8(o));
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (DGATE && j < k) {
      float s = dot[j];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) d_gate[size_t(t) * k + j] = s;
    }
  }
}

// w_t[e, i] = w[i, e]
__global__ void transpose_router_kernel(const float *__restrict__ w, int d, int E,
                                        float *__restrict__ w_t) {
  pdl_start();
  __shared__ float tile[32][33];
  const int i0 = blockIdx.x * 32, e0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + r, e = e0 + threadIdx.x;
    tile[r][threadIdx.x] = (i < d && e < E) ? w[size_t(i) * E + e] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int e = e0 + r, i = i0 + threadIdx.x;
    if (e < E && i < d) w_t[size_t(e) * d + i] = tile[threadIdx.x][r];
  }
}

// dx[t] = sum_j dx_perm[row(t,j)] + sum_j d_logits[t,j] * w_t[e_j]. HBM-bound, so what counts is how
// many warps have their k loads in flight, and that is set by the registers: 58 without the
// second sum (not ROUTER), 72 with it, 88 with it and several warps per token (SEG, few tokens). One
// kernel for all, at 88: 1,287 us instead of 1,197 at T=65536, d=7168, top-8, 66 instead of 40 at
// T=4096, top-2.
template <bool ROUTER, bool SEG>
__global__ void __launch_bounds__(kThreads) permute_bwd_kernel(
    const uint16_t *__restrict__ dx_perm, const int32_t *__restrict__ row_of_assignment,
    const int32_t *__restrict__ topk_idx, const float *__restrict__ d_logits,
    const float *__restrict__ w_t, int T, int d, int E, int k, int nseg, uint16_t *__restrict__ dx) {
  pdl_start();
  const int lane = threadIdx.x & 31;
  int t, seg;
  if (!token_segment(blockIdx.x, T, SEG ? nseg : 1, &t, &seg)) return;
  const bool router = ROUTER && d_logits != nullptr && w_t != nullptr;
  int my_row = (lane < k) ? row_of_assignment[size_t(t) * k + lane] : -1;
  int my_e = (lane < k && router) ? topk_idx[size_t(t) * k + lane] : -1;
  float my_dz = (lane < k && router) ? d_logits[size_t(t) * k + lane] : 0.f;
  int rows[8], ex[8];
  float dz[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    rows[j] = __shfl_sync(0xffffffffu, my_row, j);
    ex[j] = __shfl_sync(0xffffffffu, my_e, j);
    if (ex[j] >= E) ex[j] = -1;
    dz[j] = __shfl_sync(0xffffffffu, my_dz, j);
  }
  const int nv = d / 8, step = SEG ? 32 * nseg : 32;
  for (int c = lane + 32 * seg; c < nv; c += step) {
    uint4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < k && rows[j] >= 0) v[j] = ldg_nc_v4(dx_perm + size_t(rows[j]) * d + c * 8);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < k && rows[j] >= 0) {
        float f[8];
        unpack8(v[j], f);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] += f[q];
      }
    }
    if (router) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (j < k && ex[j] >= 0) {
          const float4 *wp = reinterpret_cast<const float4 *>(w_t + size_t(ex[j]) * d + c * 8);
          const float4 w0 = __ldg(wp), w1 = __ldg(wp + 1);
          acc[0] = fmaf(dz[j], w0.x, acc[0]); acc[1] = fmaf(dz[j], w0.y, acc[1]);
          acc[2] = fmaf(dz[j], w0.z, acc[2]); acc[3] = fmaf(dz[j], w0.w, acc[3]);
          acc[4] = fmaf(dz[j], w1.x, acc[4]); acc[5] = fmaf(dz[j], w1.y, acc[5]);
          acc[6] = fmaf(dz[j], w1.z, acc[6]); acc[7] = fmaf(dz[j], w1.w, acc[7]);
        }
      }
    }
    stg_v4(dx + size_t(t) * d + c * 8, pack8(acc));
  }
}

// Warps per token of the row kernels: one from `per_sm` warps per SM on, and with fewer tokens as
// many as give that, up to one per 32 of the row's 16-byte vectors. A lone warp's row is a chain
// of d / 256 loads' latencies: combine over 37 tokens (d 2048, top-6) 5.2 -> 2.0 us, over 191
// (d 7064, top-8) 16.2 -> 4.0 us; from ~1,000 tokens on the warps of other tokens hide it. The
// gather writes k rows per load and loses by shorter pieces sooner (T=100, d 7168: 26.8 -> 17.9
// us; T=800, d 4096: 20.9 -> 22.9 us).
constexpr int kCombineWarpsPerSm = 8, kGatherWarpsPerSm = 4;
int token_segments(int T, int d, int per_sm) {
  const int64_t warps = int64_t(moe::num_sms()) * per_sm, most = (d / 8 + 31) / 32;
  return int(std::max<int64_t>(1, std::min(most, warps / std::max(T, 1))));
}
int token_grid(int T, int nseg) { return int((int64_t(T) * nseg + kWarps - 1) / kWarps); }

// The grouped layout: group_offsets, group_counts, row_of_assignment (and token_of_row when
// given). One chunk of assignments is one launch; more take the block histograms first, and more
// than one chunk per SM their sums over the chunks. moe_permute_map, every rank block reading all
// histograms / with the sums: 16.2 / 21.8 us at 128 chunks of 256 experts, 26.4 / 22.3 at 160,
// 20.6 / 20.9 at 192 of 64, 70 / 39 at 512 of 256, 541 / 118 at 2,048. (The histogram kernel's
// blocks: 1,024 threads 38.6 us, 256 threads 39.3 at 512 chunks; 62.5 and 61.1 at 1,024.)
int launch_layout(const int32_t *idx, int64_t A, int E, int32_t *hist, const int32_t *counts,
                  int64_t rows_cap, int32_t *group_offsets, int32_t *group_counts, int32_t *row, int k,
                  int32_t *token_of_row, cudaStream_t s, const char *what) {
  const int nblk = int(std::max<int64_t>(1, (A + kChunk - 1) / kChunk));
  const bool many = nblk > moe::num_sms();
  if (nblk > 1) {
    const int threads = nblk > 4 * moe::num_sms() ? 256 : kRankThreads;
    MOE_LAUNCH("perm_hist", s, moe::launch_dep(perm_hist_kernel, nblk, threads, 0, s, idx, A, E, hist));
    if (int st = moe::launch_status(what)) return st;
  }
  if (many) {
    MOE_LAUNCH("perm_prefix", s, moe::launch_dep(perm_prefix_kernel, (E + 31) / 32, kRankThreads, 0, s, hist, E, nblk));
    if (int st = moe::launch_status(what)) return st;
  }
  auto kern = many ? perm_rank_kernel<true> : perm_rank_kernel<false>;
  MOE_LAUNCH("perm_rank", s, moe::launch_dep(kern, nblk, kRankThreads, 0, s, idx, A, E, nblk, hist, counts, rows_cap,
                                             group_offsets, group_counts, row, k, token_of_row));
  return moe::launch_status(what);
}

// The row copy into the groups and the zeroed padding rows, one launch.
int launch_gather(const uint16_t *x, const int32_t *row, int T, int d, int E, int k, int64_t rows_cap,
                  const int32_t *group_offsets, const int32_t *group_counts, uint16_t *x_perm,
                  cudaStream_t s, const char *what) {
  const int pad = E * kPadSplit, nseg = token_segments(T, d, kGatherWarpsPerSm);
  auto kern = nseg > 1 ? perm_gather_kernel<true> : perm_gather_kernel<false>;
  MOE_LAUNCH("perm_gather", s, moe::launch_dep(kern, pad + token_grid(T, nseg), kThreads, 0, s, x, row, T, d, k,
                                               nseg, rows_cap, pad, group_offsets, group_counts, x_perm));
  return moe::launch_status(what);
}

}  // namespace

namespace moe {
MOE_DEV_ERR_DEFINE_READER(permute_dev_error)
}

extern "C" {

int moe_permute(const uint16_t *x, const int32_t *topk_idx, const int32_t *counts, int T, int d,
                int E, int k, int64_t rows_cap, int32_t *group_offsets, int32_t *group_counts,
                int32_t *row_of_assignment, uint16_t *x_perm, void *ws, size_t ws_bytes,
                moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || T < 0 || d <= 0 || d % 8)
    return moe::set_error(MOE_ERR_ARG, "moe_permute: sizes T=%d d=%d E=%d k=%d", T, d, E, k);
  if (!group_offsets || !group_counts || !ws || (T > 0 && (!x || !topk_idx || !row_of_assignment || !x_perm)))
    return moe::set_error(MOE_ERR_ARG, "moe_permute: null pointer");
  if (rows_cap < moe_perm_rows_max(T, k, E))
    return moe::set_error(MOE_ERR_ARG, "moe_permute: rows_cap %lld < %lld", (long long)rows_cap,
                          (long long)moe_perm_rows_max(T, k, E));
  if (rows_cap >= (int64_t(1) << 31)) return moe::set_error(MOE_ERR_UNSUPPORTED, "moe_permute: rows_cap >= 2^31");
  if ((x && !moe::aligned16(x)) || (x_perm && !moe::aligned16(x_perm)))
    return moe::set_error(MOE_ERR_ARG, "moe_permute: x/x_perm not 16-byte aligned");
  const moe::WsLayout L = moe::ws_layout(T, d, E, k, 0);
  if (ws_bytes < L.total) return moe::set_error(MOE_ERR_WORKSPACE, "moe_permute: workspace");
  int32_t *hist = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.perm_hist);
  if (int st = launch_layout(topk_idx, int64_t(T) * k, E, hist, counts, rows_cap, group_offsets, group_counts,
                             row_of_assignment, k, nullptr, s, "moe_permute: layout"))
    return st;
  return launch_gather(x, row_of_assignment, T, d, E, k, rows_cap, group_offsets, group_counts, x_perm,
                       s, "moe_permute: gather");
}

int moe_permute_map(const int32_t *topk_idx, const int32_t *counts, int T, int E, int k,
                    int64_t rows_cap, int32_t *group_offsets, int32_t *group_counts,
                    int32_t *row_of_assignment, int32_t *token_of_row, void *ws, size_t ws_bytes,
                    moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || T < 0)
    return moe::set_error(MOE_ERR_ARG, "moe_permute_map: sizes T=%d E=%d k=%d", T, E, k);
  if (!group_offsets || !group_counts || !ws || !token_of_row ||
      (T > 0 && (!topk_idx || !row_of_assignment)))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_map: null pointer");
  if (rows_cap < moe_perm_rows_max(T, k, E))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_map: rows_cap %lld < %lld", (long long)rows_cap,
                          (long long)moe_perm_rows_max(T, k, E));
  if (rows_cap >= (int64_t(1) << 31))
    return moe::set_error(MOE_ERR_UNSUPPORTED, "moe_permute_map: rows_cap >= 2^31");
  const moe::WsLayout L = moe::ws_layout(T, 8, E, k, 0);
  if (ws_bytes < L.perm_hist + size_t(E) * std::max<int64_t>(1, (int64_t(T) * k + kChunk - 1) / kChunk) * 4)
    return moe::set_error(MOE_ERR_WORKSPACE, "moe_permute_map: workspace");
  int32_t *hist = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.perm_hist);
  if (int st = launch_layout(topk_idx, int64_t(T) * k, E, hist, counts, rows_cap, group_offsets, group_counts,
                             row_of_assignment, k, token_of_row, s, "moe_permute_map: layout"))
    return st;
  MOE_LAUNCH("pad_token", s, moe::launch_dep(pad_token_kernel, E, kThreads, 0, s, group_offsets, group_counts, E, rows_cap, token_of_row));
  return moe::launch_status("moe_permute_map: pad");
}

int moe_unpermute_combine(const uint16_t *out_perm, const int32_t *row_of_assignment,
                          const float *topk_gate, int T, int d, int k, uint16_t *y,
                          moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (k < 1 || k > 8 || T < 0 || d <= 0 || d % 8) return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine: sizes");
  if (T == 0) return MOE_OK;
  if (!out_perm || !row_of_assignment || !topk_gate || !y)
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine: null pointer");
  if (!moe::aligned16(out_perm) || !moe::aligned16(y))
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine: alignment");
  const int nseg = token_segments(T, d, kCombineWarpsPerSm);
  MOE_LAUNCH("combine", s, moe::launch_dep(combine_kernel, token_grid(T, nseg), kThreads, 0, s, out_perm, row_of_assignment, topk_gate, T, d, k, nseg, y));
  return moe::launch_status("moe_unpermute_combine: launch");
}

int moe_unpermute_combine_bwd(const uint16_t *dy, const uint16_t *out_perm,
                              const int32_t *row_of_assignment, const float *topk_gate,
                              const int32_t *group_offsets, const int32_t *group_counts, int T,
                              int d, int E, int k, uint16_t *d_out_perm, float *d_gate,
                              moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || T < 0 || d <= 0 || d % 8)
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine_bwd: sizes");
  if (!d_out_perm && !d_gate && T > 0)  // (with no tokens d_gate is empty and may be NULL)
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine_bwd: no output requested");
  if ((d_out_perm && (!group_offsets || !group_counts)) ||
      (T > 0 && (!dy || !row_of_assignment || !topk_gate || (d_gate && !out_perm))))
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine_bwd: null pointer");
  if ((d_out_perm && !moe::aligned16(d_out_perm)) || (dy && !moe::aligned16(dy)) ||
      (out_perm && !moe::aligned16(out_perm)))
    return moe::set_error(MOE_ERR_ARG, "moe_unpermute_combine_bwd: alignment");
  const int64_t rows_cap = moe_perm_rows_max(T, k, E);
  if (T == 0 && !d_out_perm) return MOE_OK;
  const int nseg = d_gate ? 1 : token_segments(T, d, kCombineWarpsPerSm);
  const int pad = d_out_perm ? E * kPadSplit : 0, grid = pad + token_grid(T, nseg);
  if (d_out_perm && d_gate) {
    MOE_LAUNCH("combine_bwd", s, moe::launch_dep(combine_bwd_kernel<true, true>, grid, kThreads, 0, s, dy, out_perm,
                                                 row_of_assignment, topk_gate, T, d, k, nseg, rows_cap, pad,
                                                 group_offsets, group_counts, d_out_perm, d_gate));
  } else if (d_out_perm) {
    MOE_LAUNCH("combine_bwd_dout", s, moe::launch_dep(combine_bwd_kernel<true, false>, grid, kThreads, 0, s, dy,
                                                      out_perm, row_of_assignment, topk_gate, T, d, k, nseg, rows_cap,
                                                      pad, group_offsets, group_counts, d_out_perm, d_gate));
  } else {
    MOE_LAUNCH("combine_bwd_dgate", s, moe::launch_dep(combine_bwd_kernel<false, true>, grid, kThreads, 0, s, dy,
                                                       out_perm, row_of_assignment, topk_gate, T, d, k, nseg, rows_cap,
                                                       pad, group_offsets, group_counts, d_out_perm, d_gate));
  }
  return moe::launch_status("moe_unpermute_combine_bwd: launch");
}

int moe_permute_bwd(const uint16_t *dx_perm, const int32_t *row_of_assignment,
                    const int32_t *topk_idx, const float *d_logits, const float *w_router, int T,
                    int d, int E, int k, uint16_t *dx, void *ws, size_t ws_bytes,
                    moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || T < 0 || d <= 0 || d % 8)
    return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: sizes");
  if (T == 0) return MOE_OK;
  if (!dx_perm || !row_of_assignment || !dx) return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: null pointer");
  if ((d_logits == nullptr) != (w_router == nullptr))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: d_logits and w_router go together");
  if (!moe::aligned16(dx_perm) || !moe::aligned16(dx)) return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: alignment");
  float *w_t = nullptr;
  if (w_router) {
    if (!topk_idx || !ws) return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: router term needs topk_idx and ws");
    const moe::WsLayout L = moe::ws_layout(T, d, E, k, 0);
    if (ws_bytes < L.total) return moe::set_error(MOE_ERR_WORKSPACE, "moe_permute_bwd: workspace");
    if (!moe::aligned16(ws)) return moe::set_error(MOE_ERR_ARG, "moe_permute_bwd: ws alignment");
    w_t = reinterpret_cast<float *>(static_cast<char *>(ws) + L.w_router_t);
    dim3 grid((d + 31) / 32, (E + 31) / 32), block(32, 8);
    MOE_LAUNCH("transpose_router", s, moe::launch_dep(transpose_router_kernel, grid, block, 0, s, w_router, d, E, w_t));
    if (int st = moe::launch_status("moe_permute_bwd: transpose")) return st;
  }
  const int nseg = token_segments(T, d, kCombineWarpsPerSm);
  auto kern = d_logits && w_t ? (nseg > 1 ? permute_bwd_kernel<true, true> : permute_bwd_kernel<true, false>)
                              : (nseg > 1 ? permute_bwd_kernel<false, true> : permute_bwd_kernel<false, false>);
  MOE_LAUNCH("permute_bwd", s, moe::launch_dep(kern, token_grid(T, nseg), kThreads, 0, s, dx_perm,
                                               row_of_assignment, topk_idx, d_logits, w_t, T, d, E, k, nseg, dx));
  return moe::launch_status("moe_permute_bwd: launch");
}

}  // extern "C"

// ---------------------------------------------------------------------------
// moe_permute_noalloc: moe_permute for callers that cannot allocate device
// memory (no cudaMalloc and no caller workspace), e.g. an inference engine's
// plugin, whose device memory the engine planned and owns before execution
// and which receives only its input and output buffers. The
// per-block histograms live in a fixed array compiled into the library
// instead of the caller's workspace.
//
// The array holds kNoAllocScratchInts int32 entries (256 KiB). A call needs
// E * ceil(T*k / 4096) of them, so 256 experts fit with up to 1,048,576
// assignments (T*k). Every GPU that loads the library keeps the array until
// the process exits. All calls share it: calls whose kernels overlap on the
// GPU (different streams, or different host threads) race on it and must be
// serialized by the caller. Nothing in it has to start at zero: every entry a
// call reads was written earlier in the same call.
constexpr int kNoAllocScratchInts = 65536;
static __device__ __align__(256) int32_t g_perm_noalloc_scratch[kNoAllocScratchInts];

namespace {
typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);

// Unique id of the calling thread's current CUDA context (0: none is current yet).
// Ids are never reused, so a context created after cudaDeviceReset, or another
// context of the same device, has an id of its own.
int current_context_id(unsigned long long *id) {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<CtxGetCurrentFn>(p);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess && q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<CtxGetIdFn>(p);
  });
  if (!get_current || !get_id)
    return moe::set_error(MOE_ERR_CUDA, "moe_permute_noalloc: cuCtxGetCurrent/cuCtxGetId unavailable");
  CUcontext ctx = nullptr;
  if (get_current(&ctx) != CUDA_SUCCESS)
    return moe::set_error(MOE_ERR_CUDA, "moe_permute_noalloc: cuCtxGetCurrent failed");
  *id = 0;
  if (ctx && get_id(ctx, id) != CUDA_SUCCESS)
    return moe::set_error(MOE_ERR_CUDA, "moe_permute_noalloc: cuCtxGetId failed");
  return MOE_OK;
}

// Device address of the array in the current context. Host code cannot use the
// array's name as a device pointer, and the address belongs to the context that
// loaded the library's module: it is looked up once per context (keyed by the
// context's unique id) and cached; another context of the same device, or the new
// primary context after cudaDeviceReset, gets a lookup of its own.
int noalloc_scratch(int32_t **out) {
  constexpr int kSlots = 64;
  static std::mutex mu;
  static unsigned long long ids[kSlots] = {0};
  static int32_t *addr[kSlots] = {nullptr};
  static int next = 0;
  unsigned long long id = 0;
  if (int st = current_context_id(&id)) return st;
  std::lock_guard<std::mutex> g(mu);
  if (id != 0) {
    for (int i = 0; i < kSlots; ++i)
      if (ids[i] == id) {
        *out = addr[i];
        return MOE_OK;
      }
  }
  void *p = nullptr;  // the runtime makes the primary context current if none is
  cudaError_t e = cudaGetSymbolAddress(&p, g_perm_noalloc_scratch);
  if (e != cudaSuccess) return moe::cuda_status(e, "moe_permute_noalloc: cudaGetSymbolAddress");
  if (id == 0 && (current_context_id(&id) != MOE_OK || id == 0))
    return moe::set_error(MOE_ERR_CUDA, "moe_permute_noalloc: no current context");
  ids[next] = id;  // oldest entry replaced when all slots are taken
  addr[next] = static_cast<int32_t *>(p);
  next = (next + 1) % kSlots;
  *out = static_cast<int32_t *>(p);
  return MOE_OK;
}
}  // namespace

extern "C" int moe_permute_noalloc(const uint16_t *x, const int32_t *topk_idx,
                                   const int32_t *counts, int T, int d, int E, int k,
                                   int64_t rows_cap, int32_t *group_offsets,
                                   int32_t *group_counts, int32_t *row_of_assignment,
                                   uint16_t *x_perm, moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || T < 0 || d <= 0 || d % 8)
    return moe::set_error(MOE_ERR_ARG, "moe_permute_noalloc: sizes T=%d d=%d E=%d k=%d", T, d, E, k);
  const int64_t A = int64_t(T) * k;
  const int64_t nblk64 = std::max<int64_t>(1, (A + kChunk - 1) / kChunk);
  if (int64_t(E) * nblk64 > kNoAllocScratchInts)
    return moe::set_error(MOE_ERR_UNSUPPORTED,
                          "moe_permute_noalloc: E * ceil(T*k/%d) = %lld exceeds the built-in "
                          "scratch of %d entries (use moe_permute with a workspace)",
                          kChunk, (long long)(int64_t(E) * nblk64), kNoAllocScratchInts);
  if (!group_offsets || !group_counts || (T > 0 && (!x || !topk_idx || !row_of_assignment || !x_perm)))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_noalloc: null pointer");
  if (rows_cap < moe_perm_rows_max(T, k, E))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_noalloc: rows_cap %lld < %lld",
                          (long long)rows_cap, (long long)moe_perm_rows_max(T, k, E));
  if (rows_cap >= (int64_t(1) << 31))
    return moe::set_error(MOE_ERR_UNSUPPORTED, "moe_permute_noalloc: rows_cap >= 2^31");
  if ((x && !moe::aligned16(x)) || (x_perm && !moe::aligned16(x_perm)))
    return moe::set_error(MOE_ERR_ARG, "moe_permute_noalloc: x/x_perm not 16-byte aligned");
  int32_t *hist = nullptr;
  if (int st = noalloc_scratch(&hist)) return st;
  if (int st = launch_layout(topk_idx, A, E, hist, counts, rows_cap, group_offsets, group_counts,
                             row_of_assignment, k, nullptr, s, "moe_permute_noalloc: layout"))
    return st;
  return launch_gather(x, row_of_assignment, T, d, E, k, rows_cap, group_offsets, group_counts, x_perm,
                       s, "moe_permute_noalloc: gather");
}
