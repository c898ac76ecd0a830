// Router (fp32 logits, top-k, softmax over the selected experts, histogram),
// the standalone histogram, and the router backward.
//
// Routing indicator E[i,j,l] and per-expert token number: Sec. 3.2, Eq. 1 and
// Algorithm 1 Step 1 of the LAEP paper. Pruned experts receive no token
// (Sec. 4, Table 5): their logit is -inf before the top-k.
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "tmap.cuh"

MOE_DEV_ERR_DECL

namespace {

constexpr int kTopkThreads = 128;
int padded_experts(int E) { return E <= 64 ? 64 : (E <= 128 ? 128 : (E <= 192 ? 192 : 256)); }

__global__ void zero_i32_kernel(int32_t *p, int n) {
  pdl_start();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0;
}

// ---- logits on the tensor cores ----------------------------------------------
// The fp32 router weight is split into three bf16 terms, W = W_hi + W_mid + W_lo,
// each the bf16 rounding of what the earlier terms leave (the bf16x3 scheme of
// Henry, Tang and Heinecke, "Leveraging the bfloat16 artificial intelligence
// datatype for higher-precision computations", 2019). Three 8-bit significands
// cover the 24 of a normal fp32 weight, every bf16 x bf16 product is exact in
// fp32 and accumulates in fp32 in tensor memory, so the logits carry fp32
// accumulation error only.
//
// One CTA = one or two 128-token tiles x one range of k-blocks (a split of the
// reduction over d when there are fewer tiles than CTA slots). Warp 0 issues the
// TMA loads (x tile + the three weight terms per k-block), warp 1 owns TMEM and
// issues the MMAs, then all four warps read the accumulator (one TMEM lane
// quarter each) and write the partial logits partial[split][t][0..NP). The same
// kernel computes the router weight gradient with the roles changed (see
// route_tc_kernel): 128-feature tiles of x^T, the reduction over tokens.
constexpr int kRtBM = 128;       // tokens per tile (TMEM lanes)
constexpr int kRtBK = 64;        // k-block: 64 bf16 = one 128-byte swizzle row
constexpr int kRtThreads = 128;
constexpr int kRtSms = 152;           // SMs of a GB300: the splits aim to fill them
constexpr int kRtSmemPerSm = 233472;  // shared memory per SM (228 KB)
constexpr int kRtLogitsSplits = 8;
constexpr int kRtDwSplits = 64;
constexpr uint32_t kRtABytes = kRtBM * kRtBK * 2;
constexpr int kRtMaxSmem = 232448;  // opt-in dynamic shared memory per CTA
constexpr uint64_t kRtWaitNs = 2000000000ull;

struct RouteTcParams {
  int M;             // output rows: tokens (logits) or d_model (router weight gradient)
  int MT;            // 128-row tiles per CTA (1 or 2); tile m's accumulator at TMEM column 256*m
  int kb_per_split;  // k-blocks of one split
  int nkb;           // k-blocks of the reduction (over d, or over the padded tokens)
  int NP;            // experts rounded up to 16
  int NE;            // row stride of the partial logits
  int stages;        // shared-memory ring depth
  uint32_t tmem_cols;
  float *partial;
};

// Experts rounded up to the MMA's N granularity, and the matching TMEM allocation.
int route_tc_np(int E) { return (E + 15) / 16 * 16; }
// Terms of the second operand (the weight, or dZ) per MMA. Logits: 1, each k-step adds the hi, mid
// and lo products to one accumulator. x^T dZ: as many as fit along N (256), each with an accumulator of
// its own, added at the end; the x tile is then read from shared memory once (up to 80 experts)
// or twice (up to 128) per k-step instead of three times, and shared memory sets the pace of
// these short-N MMAs: 43 / 31 us at T=16384, d=4096, 64 experts, 47 / 40 us at T=35700, d=2856, 57.
// At least one: the workspace is also sized for expert counts that moe_route and moe_route_bwd
// refuse (E > 256), and the plan divides by this.
int route_dw_group(int NP) { return std::max(1, std::min(3, 256 / NP)); }
uint32_t route_tc_tmem_cols(int c, int MT) {  // c: accumulator columns of one tile
  if (MT == 2) return 512u;
  return c <= 32 ? 32u : (c <= 64 ? 64u : (c <= 128 ? 128u : 256u));
}
uint32_t route_tc_stage_bytes(int NP, int MT) { return uint32_t(MT) * kRtABytes + 3u * uint32_t(NP) * 128u; }
size_t route_tc_smem(int NP, int stages, int MT) {
  return 1024 + size_t(stages) * route_tc_stage_bytes(NP, MT) + size_t(2 * stages + 1) * 8 + 16;
}
// CTAs per SM and ring depth: with one 128-row tile per CTA, two CTAs per SM if a ring of at
// least two stages each fits (more independent x streams per SM: measured faster than one
// CTA with a deeper ring); else one with the deepest ring that fits (0 stages: none of two).
void route_tc_ring(int NP, int MT, int *per_sm, int *stages) {
  *per_sm = MT == 1 && 2 * (route_tc_smem(NP, 2, 1) + 1024) <= size_t(kRtSmemPerSm) ? 2 : 1;
  int st = 0;
  while (st < 8 && (*per_sm == 2 ? 2 * (route_tc_smem(NP, st + 1, 1) + 1024) <= size_t(kRtSmemPerSm)
                                 : int64_t(st + 1) * route_tc_stage_bytes(NP, MT) <= kRtMaxSmem - 2048))
    ++st;
  *stages = st >= 2 ? st : 0;
}

struct RtPlan {
  int MT;  // 128-row tiles per CTA
  int stages, splits, kb_per_split;
};
// Logits, M tokens over K = d. Two tiles per CTA from 97 to 192 experts, where the three weight
// terms of a k-block (3 x NP x 128 bytes) outweigh the 16 KB x tile: two x tiles share each
// weight stage. Splits: enough CTAs to fill the SMs' CTA slots when the tokens give few tiles. The
// plan fixes the order in which a logit's products are summed, and with it the last bits that
// decide a near tie: it is a function of (M, K, NP) alone, and a change of it can route a token
// differently.
RtPlan route_logits_plan(int M, int K, int NP) {
  RtPlan r;
  int per_sm;
  r.MT = NP > 96 && NP <= 192 ? 2 : 1;
  route_tc_ring(NP, r.MT, &per_sm, &r.stages);
  const int rows = kRtBM * r.MT, tiles = std::max(1, (M + rows - 1) / rows);
  const int nkb = (K + kRtBK - 1) / kRtBK;
  const int s = std::max(1, std::min({kRtSms * per_sm / tiles, kRtLogitsSplits, nkb}));
  r.kb_per_split = (nkb + s - 1) / s;
  r.splits = (nkb + r.kb_per_split - 1) / r.kb_per_split;  // every split gets at least one k-block
  return r;
}
// x^T dZ, M = d features over K tokens: the tiles per CTA and splits of the reduction with the
// least estimated time (ns). An SM takes a k-block of a CTA in the longest of its share of the HBM
// rate for the x tiles, its shared-memory traffic (TMA writes, MMA reads) at ~243 B/ns, and, with
// few CTAs, a load's way through the ring (~2.3 us for load, wait and MMA over the stages); a
// split adds its partial sums' write and read. A function of (M, K, NP) alone, so the workspace
// size is too. K > 0. Measured, with the logits' plan (at most 8 splits) / with this one: 30 /
// 12.6 us at T=22360, d=1128, 28 experts (9 tiles: 72 CTAs / 32 splits), 67 / 40 us at T=35700,
// d=2856, 57 experts, 22.9 / 18.0 us at T=3516, d=3328, 167 experts; both 49 us at T=8191, d=7168, 171.
RtPlan route_dw_plan(int M, int K, int NP) {
  const int nkb = (K + kRtBK - 1) / kRtBK;
  const int group = route_dw_group(NP), mmas = (3 + group - 1) / group;
  const int64_t ne = (NP + 31) / 32 * 32;
  RtPlan best{1, 2, 1, nkb};
  int64_t best_ns = INT64_MAX;
  for (int mt = 1; mt <= (M > kRtBM ? 2 : 1); ++mt) {
    int per_sm, stages;
    route_tc_ring(NP, mt, &per_sm, &stages);
    if (stages == 0) continue;
    const int64_t tiles = std::max(1, (M + kRtBM * mt - 1) / (kRtBM * mt));
    const int64_t a = int64_t(mt) * kRtABytes, w = int64_t(3) * NP * 128;
    const int64_t busy = std::max<int64_t>(a * 1000 / 44700, (a + w + mmas * a + mt * w) * 1000 / 243000);
    const int64_t ring = 2300 / stages, slots = int64_t(kRtSms) * per_sm;
    for (int s = 1; s <= std::min(nkb, kRtDwSplits); ++s) {
      const int per = (nkb + s - 1) / s;
      if ((nkb + per - 1) / per != s) continue;  // every split gets at least one k-block
      const int64_t full = tiles * s / slots, rest = tiles * s % slots;
      int64_t ns = full * (per * std::max(per_sm * busy, ring) + 1500);
      if (rest > 0) ns += per * std::max(rest > kRtSms ? 2 * busy : busy, ring) + 1500;
      if (s > 1) ns += s * int64_t(M) * ne * 8 / 4000;
      if (ns < best_ns) {
        best_ns = ns;
        best = {mt, stages, s, per};
      }
    }
  }
  return best;
}

// Router weight gradient: tokens padded to one k-block, and the row stride of its
// partial sums (the epilogue writes 32 columns at a time).
int route_tokens_padded(int T) { return (T + kRtBK - 1) / kRtBK * kRtBK; }
int route_dw_stride(int E) { return (route_tc_np(E) + 31) / 32 * 32; }

// W [d, E] fp32 -> W3 [3][NP][d] bf16 (hi, mid, lo; rows e >= E are zero), by
// 32 x 32 tiles transposed through shared memory. The first blocks also zero the counts that
// the top-k kernel adds to (nullptr: none).
__global__ void route_split_w_kernel(const float *__restrict__ w, int d, int E, int NP,
                                     uint16_t *__restrict__ w3, int32_t *__restrict__ counts) {
  __shared__ float tile[32][33];
  pdl_start();
  if (counts != nullptr && blockIdx.x == 0 && threadIdx.y == 0 && blockIdx.y * 32 + threadIdx.x < E)
    counts[blockIdx.y * 32 + threadIdx.x] = 0;
  const int k0 = blockIdx.x * 32, e0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int i = ty; i < 32; i += 8) {
    const int k = k0 + i, e = e0 + tx;
    tile[i][tx] = (k < d && e < E) ? w[size_t(k) * E + e] : 0.f;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int e = e0 + i, k = k0 + tx;
    if (e < NP && k < d) {
      const float v = tile[tx][i];
      const __nv_bfloat16 hi = __float2bfloat16_rn(v);
      const float r1 = v - __bfloat162float(hi);
      const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
      const float r2 = r1 - __bfloat162float(mid);
      const __nv_bfloat16 lo = __float2bfloat16_rn(r2);
      const size_t plane = size_t(NP) * d, at = size_t(e) * d + k;
      w3[at] = __bfloat16_as_ushort(hi);
      w3[plane + at] = __bfloat16_as_ushort(mid);
      w3[2 * plane + at] = __bfloat16_as_ushort(lo);
    }
  }
}

// DW = false: the logits, partial[split][t][e] = x[t, k-range] . W3[e, k-range].
// DW = true: the router weight gradient, partial[split][i][e] = sum over the split's
// tokens t of x[t, i] * dZ[t, e] (A = x^T, read MN-major from x itself as two 64 x 64
// boxes per k-block; B = dZ's three bf16 terms, K-major [3][NP][T padded to 64]).
// G = terms per MMA (see route_dw_group), at compile time: the issuing thread's loop sets the pace
// otherwise (with a bound read from the parameters 110 instead of 79 us at T=32768, 128 experts).
// AHEAD (logits): a stage's next x tile goes to L2 while this one loads (see launch_route_tc).
template <bool DW, int G, bool AHEAD>
__global__ void __launch_bounds__(kRtThreads, 1)
    route_tc_kernel(const __grid_constant__ CUtensorMap tmX,
                    const __grid_constant__ CUtensorMap tmW, const RouteTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = tc::smem_u32(smem_raw);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  const uint32_t b_bytes = uint32_t(p.NP) * 128u;
  const uint32_t a_bytes = uint32_t(p.MT) * kRtABytes;  // the CTA's x tiles of a k-block
  const uint32_t stage_bytes = a_bytes + 3u * b_bytes;
  const int S = p.stages;
  const uint32_t s0 = raw + pad;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw + pad + size_t(S) * stage_bytes);
  int *misc = reinterpret_cast<int *>(bars + 2 * S + 1);
  volatile int *abort_flag = misc + 1;
  volatile int no_abort = 0;
  const uint32_t bar0 = tc::smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (S + s); };
  const uint32_t done_bar = bar0 + 8u * (2 * S);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mt = blockIdx.x, split = blockIdx.y;
  const int kb0 = split * p.kb_per_split, nk = min(p.nkb, kb0 + p.kb_per_split) - kb0;
  // Each token tile starts its k-loop at its own offset, so that the CTAs do not all read
  // the same weight tile from L2 at the same time (the order is fixed per tile; without it
  // 88 instead of 71 us at T=26750, d=4296, 61 experts). x^T dZ's feature tiles read slices
  // of the same token rows and stay in step (48 against 51 us at T=35700, d=2856).
  const int rot = !DW && nk > 0 ? int((mt * 7u) % uint32_t(nk)) : 0;
  const uint32_t idesc_g = tc::idesc_bf16_f32(kRtBM, G * p.NP, DW, false);
  const uint32_t idesc_1 = tc::idesc_bf16_f32(kRtBM, p.NP, DW, false);

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(full_bar(s), 1);
      tc::mbar_init(empty_bar(s), 1);
    }
    tc::mbar_init(done_bar, 1);
    tc::fence_mbar_init();
    misc[1] = 0;
  }
  if (warp == 0 && lane == 0) {
    tc::tma_prefetch_desc(&tmX);
    tc::tma_prefetch_desc(&tmW);
  }
  if (warp == 1) {
    tc::tmem_alloc(tc::smem_u32(misc), p.tmem_cols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem_base = static_cast<uint32_t>(misc[0]);
  pdl_start();  // TMEM is allocated; set-up overlaps the end of the previous kernel

  if (warp == 0 && lane == 0) {
    // ---- TMA producer ----
    uint32_t it = 0;
    for (; int(it) < nk; ++it) {
      const int kb = kb0 + (int(it) + rot) % nk;
      const int s = it % S;
      const uint32_t ph = (it / S) & 1u;
      if (!tc::mbar_wait(empty_bar(s), ph ^ 1u, kRtWaitNs, abort_flag)) {
        dev_flag(&g_dev_err, MOE_DEV_WAIT_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      tc::mbar_arrive_expect_tx(full_bar(s), stage_bytes);
      const uint32_t dst = s0 + s * stage_bytes;
      const int k0 = kb * kRtBK;
      for (int m = 0; m < p.MT; ++m) {
        const int row0 = (mt * p.MT + m) * kRtBM;
        const uint32_t am = dst + uint32_t(m) * kRtABytes;
        if (DW) {  // x^T: features row0 .. +127 (two 64-wide boxes) x tokens k0 .. k0+63
          tc::tma_load_2d(am, &tmX, full_bar(s), row0, k0);
          tc::tma_load_2d(am + 64 * 128, &tmX, full_bar(s), row0 + 64, k0);
        } else {
          tc::tma_load_2d(am, &tmX, full_bar(s), k0, row0);
        }
      }
#pragma unroll
      for (int j = 0; j < 3; ++j)
        tc::tma_load_2d(dst + a_bytes + j * b_bytes, &tmW, full_bar(s), k0, j * p.NP);
      if (AHEAD && int(it) + 2 < nk) {
        const int k2 = (kb0 + (int(it) + 2 + rot) % nk) * kRtBK;
        for (int m = 0; m < p.MT; ++m) {
          const int row0 = (mt * p.MT + m) * kRtBM;
          if (row0 < p.M) tc::tma_prefetch_2d(&tmX, k2, row0);
        }
      }
    }
    // every issued load lands before the CTA may exit (also after an abort)
    for (int s = 0; s < S; ++s) {
      if (it > uint32_t(s)) {
        const uint32_t n = (it - 1 - s) / S;
        if (!tc::mbar_wait(full_bar(s), n & 1u, kRtWaitNs, &no_abort))
          dev_flag(&g_dev_err, MOE_DEV_WAIT_TIMEOUT);
      }
    }
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer ----
    uint32_t it = 0;
    bool issued = false;
    for (; int(it) < nk; ++it) {
      const int s = it % S;
      const uint32_t ph = (it / S) & 1u;
      if (!tc::mbar_wait(full_bar(s), ph, kRtWaitNs, abort_flag)) {
        dev_flag(&g_dev_err, MOE_DEV_WAIT_TIMEOUT);
        *abort_flag = 1;
        break;
      }
      tc::fence_after_sync();
      const uint32_t a_s = s0 + s * stage_bytes, b_s = a_s + a_bytes;
      // (a descriptor's address field counts 16 bytes: steps are plain additions)
      const uint64_t b0 = tc::smem_desc_sw128(b_s, 16, 1024);
      for (int m = 0; m < p.MT; ++m) {
        const uint32_t am = a_s + uint32_t(m) * kRtABytes, d = tmem_base + uint32_t(m) * 256u;
        const uint64_t a0 = DW ? tc::smem_desc_sw128(am, 8192, 1024) : tc::smem_desc_sw128(am, 16, 1024);
#pragma unroll
        for (int kk = 0; kk < kRtBK / 16; ++kk) {
          const uint64_t ad = a0 + uint64_t(DW ? kk * 128 : kk * 2);
          tc::mma_bf16(d, ad, b0 + uint64_t(kk * 2), idesc_g, (it != 0 || kk != 0) ? 1u : 0u);
#pragma unroll
          for (int j = G; j < 3; ++j)  // terms that did not fit: into the first accumulator
            tc::mma_bf16(d, ad, b0 + uint64_t(kk * 2) + uint64_t(j) * (b_bytes >> 4), idesc_1, 1u);
        }
      }
      tc::mma_commit(empty_bar(s));
      issued = true;
    }
    if (issued) tc::mma_commit(done_bar);
    else *abort_flag = 1;  // nothing to wait for: the epilogue must not wait either
  }
  __syncwarp();

  // ---- epilogue: TMEM lane quarter `warp` -> 32 output rows x NP partial sums ----
  int ok = 0;
  if (lane == 0) {
    ok = tc::mbar_wait(done_bar, 0, kRtWaitNs, abort_flag) ? 1 : 0;
    if (!ok && !*abort_flag) {
      dev_flag(&g_dev_err, MOE_DEV_WAIT_TIMEOUT);
      *abort_flag = 1;
    }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok) {
    tc::fence_after_sync();
    for (int m = 0; m < p.MT; ++m) {
      const int t = (mt * p.MT + m) * kRtBM + warp * 32 + lane;
      float *dst = p.partial + (size_t(split) * p.M + t) * p.NE;
      for (int c0 = 0; c0 < p.NP; c0 += 32) {
        uint32_t r[32];
        const uint32_t tb = tmem_base + (uint32_t(warp * 32) << 16) + uint32_t(m) * 256u + uint32_t(c0);
        tc::tmem_ld_32x32b_x32(tb, r);
        tc::tmem_ld_wait();
#pragma unroll
        for (int j = 1; j < G; ++j) {
          uint32_t q[32];
          tc::tmem_ld_32x32b_x32(tb + uint32_t(j * p.NP), q);
          tc::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(q[i]));
        }
        if (t < p.M) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            stg_v4(dst + c0 + 4 * q, make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]));
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

// The K largest (key, expert) pairs so far, descending; equal keys by ascending expert.
template <int K> struct TopList {
  unsigned key[K];  // order-preserving key of a logit, 0: empty
  int e[K];
  __device__ __forceinline__ TopList() {
#pragma unroll
    for (int s = 0; s < K; ++s) {
      key[s] = 0u;
      e[s] = -1;
    }
  }
  // Experts come in ascending order: a later one passes strictly smaller keys only (the
  // entries from there on move down one slot).
  __device__ __forceinline__ void add(unsigned x, int xe) {
    bool up = false;
#pragma unroll
    for (int s = 0; s < K; ++s) {
      up = up || x > key[s];
      const unsigned lk = up ? key[s] : x;
      const int le = up ? e[s] : xe;
      key[s] = up ? x : key[s];
      e[s] = up ? xe : e[s];
      x = lk;
      xe = le;
    }
  }
  static __device__ __forceinline__ bool before(unsigned ka, int ea, unsigned kb, int eb) {
    return ka > kb || (ka == kb && ea < eb);
  }
  // The K largest of this list and lane ^ `lane_xor`'s: the larger of entry s here and entry
  // K-1-s there are those K, as a bitonic sequence, which log2(K) exchange stages sort.
  __device__ __forceinline__ void merge(int lane_xor) {
    unsigned ok[K];
    int oe[K];
#pragma unroll
    for (int s = 0; s < K; ++s) {
      ok[s] = __shfl_xor_sync(0xffffffffu, key[s], lane_xor);
      oe[s] = __shfl_xor_sync(0xffffffffu, e[s], lane_xor);
    }
#pragma unroll
    for (int s = 0; s < K; ++s) {
      const bool other = before(ok[K - 1 - s], oe[K - 1 - s], key[s], e[s]);
      key[s] = other ? ok[K - 1 - s] : key[s];
      e[s] = other ? oe[K - 1 - s] : e[s];
    }
#pragma unroll
    for (int h = K / 2; h > 0; h >>= 1)
#pragma unroll
      for (int s = 0; s < K; ++s)
        if ((s & h) == 0) {
          const bool sw = before(key[s + h], e[s + h], key[s], e[s]);
          const unsigned ka = key[s], kb = key[s + h];
          const int ea = e[s], eb = e[s + h];
          key[s] = sw ? kb : ka;
          e[s] = sw ? eb : ea;
          key[s + h] = sw ? ka : kb;
          e[s + h] = sw ? ea : eb;
        }
  }
};

// LPT (4 or 16) lanes per token: logits = sum of the split partials (fixed order) + bias, pruned
// experts -inf; top-k (ties to the lower index), softmax over the selected logits,
// per-expert histogram (shared per block, then one global add per expert and block).
// Lane q keeps the K largest logits of experts 4 LPT i + 4 q .. + 3 in registers (~5 K
// instructions per logit, 32 / LPT tokens per instruction), exchanges merge the lists.
// Issue-bound with many tokens: 4 lanes, ~250 warp instructions per token at 128 experts, top-8,
// against ~1,000 for a warp per token with two redux per selected expert: 21 us instead of 40
// at T=32768 (the compares and selects, at half the issue rate, are its bound now). Latency-bound
// with few: 16 lanes, a quarter of the chain per lane.
template <int K, int LPT>
__global__ void __launch_bounds__(kTopkThreads) route_topk_kernel(
    const float *__restrict__ partial, int splits, int NE, const float *__restrict__ logits_in,
    const float *__restrict__ bias, const uint8_t *__restrict__ active_mask, int T, int E, int k,
    float *__restrict__ logits_out, int32_t *__restrict__ topk_idx, float *__restrict__ topk_gate,
    int32_t *__restrict__ counts) {
  __shared__ int hist[256];
  __shared__ __align__(16) float s_bias[256];
  __shared__ uint8_t s_live[256];
  const int tid = threadIdx.x, q = tid % LPT;
  for (int e = tid; e < 256; e += kTopkThreads) hist[e] = 0;
  pdl_start();
  for (int e = tid; e < 256; e += kTopkThreads) {
    s_bias[e] = (bias != nullptr && e < E) ? bias[e] : 0.f;
    s_live[e] = e < E && (active_mask == nullptr || active_mask[e] != 0);
  }
  __syncthreads();
  constexpr int per_block = kTopkThreads / LPT;
  // (whole warps stay in the loop: the merges are warp-wide)
  for (int t0 = blockIdx.x * per_block; t0 < T; t0 += gridDim.x * per_block) {
    const int t = t0 + tid / LPT;
    const bool mine = t < T;
    TopList<K> top;
    // four chunks of four experts at a time, so that their loads (of up to four partials each)
    // are in flight together
    for (int g0 = 0; g0 < E; g0 += 16 * LPT) {
      float z[4][4] = {};
      if (mine) {
        if (logits_in != nullptr) {
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int e = g0 + 4 * (c * LPT + q) + i;
              if (e < E) z[c][i] = logits_in[size_t(t) * E + e];
            }
        } else {
          const float *src = partial + size_t(t) * NE + g0 + 4 * q;
          const size_t plane = size_t(T) * NE;
          for (int y0 = 0; y0 < splits; y0 += 4) {  // summed in order
            float4 v[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int c = 0; c < 4; ++c)
                if (y0 + u < splits && g0 + 4 * (c * LPT + q) < E)
                  v[u][c] = *reinterpret_cast<const float4 *>(src + (y0 + u) * plane + 4 * LPT * c);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int c = 0; c < 4; ++c)
                if (y0 + u < splits && g0 + 4 * (c * LPT + q) < E) {
                  z[c][0] += v[u][c].x;
                  z[c][1] += v[u][c].y;
                  z[c][2] += v[u][c].z;
                  z[c][3] += v[u][c].w;
                }
          }
        }
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int e0 = g0 + 4 * (c * LPT + q);
        if (e0 < E) {
          if (logits_in == nullptr && bias != nullptr) {
            const float4 b = *reinterpret_cast<const float4 *>(s_bias + e0);
            z[c][0] += b.x;
            z[c][1] += b.y;
            z[c][2] += b.z;
            z[c][3] += b.w;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int e = e0 + i;
            float v = z[c][i];
            if (!s_live[e]) v = -INFINITY;
            if (e < E) {
              if (logits_out != nullptr && mine) logits_out[size_t(t) * E + e] = v;
              // a larger float gives a larger key; -0 is taken as +0 so that equal logits tie
              const unsigned u = __float_as_uint(v == 0.f ? 0.f : v);
              top.add((u & 0x80000000u) ? ~u : (u | 0x80000000u), e);
            }
          }
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int h = 1; h < LPT; h <<= 1) top.merge(h);
    if (!mine) continue;
    // softmax over the selected logits (renormalised top-k), fp32
    float ex[K], den = 0.f, zmax = 0.f;
    bool too_few = false;
#pragma unroll
    for (int s = 0; s < K; ++s) {
      if (s < k) {
        const unsigned m = top.key[s];
        const float v = __uint_as_float((m & 0x80000000u) ? (m & 0x7fffffffu) : ~m);
        if (s == 0) zmax = v;
        ex[s] = expf(v - zmax);
        den += ex[s];
        if (v == -INFINITY) too_few = true;
      }
    }
    if (q == 0 && too_few) dev_flag(&g_dev_err, MOE_DEV_TOO_FEW_LIVE);
#pragma unroll
    for (int s = 0; s < K; ++s) {
      if (s < k && s % LPT == q) {
        topk_idx[size_t(t) * k + s] = top.e[s];
        topk_gate[size_t(t) * k + s] = ex[s] / den;
        if (top.e[s] >= 0) atomicAdd(&hist[top.e[s]], 1);
      }
    }
  }
  __syncthreads();
  if (counts != nullptr)
    for (int e = tid; e < E; e += kTopkThreads)
      if (hist[e]) atomicAdd(&counts[e], hist[e]);
}

// store: the only block of the launch, which writes the counts instead of adding to them.
__global__ void load_stats_kernel(const int32_t *__restrict__ topk_idx, int64_t A, int E, int store,
                                  int32_t *__restrict__ counts) {
  __shared__ int hist[256];
  for (int e = threadIdx.x; e < E; e += blockDim.x) hist[e] = 0;
  __syncthreads();
  pdl_start();
  for (int64_t a = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; a < A;
       a += int64_t(gridDim.x) * blockDim.x) {
    const int e = topk_idx[a];
    if (e >= 0 && e < E)
      atomicAdd(&hist[e], 1);
    else
      dev_flag(&g_dev_err, MOE_DEV_BAD_EXPERT);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += blockDim.x) {
    if (store) counts[e] = hist[e];
    else if (hist[e]) atomicAdd(&counts[e], hist[e]);
  }
}

// ---- router backward -------------------------------------------------------

// Softmax backward over the selected k, d_logits[t,j] = g_j (dg_j - sum_i g_i dg_i),
// and dZ (the [T, E] logit gradient, zero off the selected experts) as three bf16
// terms, K-major for the tensor cores: dz3[s][e][t] for e < NP, t < Tp (tokens padded
// to 64; the padding is zero). One thread per token and 16 experts (blockIdx.y); the
// y = 0 blocks also write d_logits.
constexpr int kDzExperts = 16;
__global__ void route_bwd_dz_kernel(const int32_t *__restrict__ topk_idx,
                                    const float *__restrict__ gate, const float *__restrict__ dgate,
                                    int T, int Tp, int k, int NP, float *__restrict__ d_logits,
                                    uint16_t *__restrict__ dz3) {
  pdl_start();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Tp) return;
  float g[8], dg[8], s = 0.f;
  int ei[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    g[j] = 0.f;
    dg[j] = 0.f;
    ei[j] = -1;
    if (j < k && t < T) {
      g[j] = gate[size_t(t) * k + j];
      dg[j] = dgate[size_t(t) * k + j];
      ei[j] = topk_idx[size_t(t) * k + j];
      s = fmaf(g[j], dg[j], s);
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    g[j] = g[j] * (dg[j] - s);
    if (blockIdx.y == 0 && j < k && t < T) d_logits[size_t(t) * k + j] = g[j];
  }
  const size_t plane = size_t(NP) * Tp;
  const int e0 = blockIdx.y * kDzExperts;
  for (int e = e0; e < min(NP, e0 + kDzExperts); ++e) {
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (ei[j] == e) v = g[j];  // the k selected experts of a token are distinct
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(mid);
    const __nv_bfloat16 lo = __float2bfloat16_rn(r2);
    const size_t at = size_t(e) * Tp + t;
    dz3[at] = __bfloat16_as_ushort(hi);
    dz3[plane + at] = __bfloat16_as_ushort(mid);
    dz3[2 * plane + at] = __bfloat16_as_ushort(lo);
  }
}

// dw_router[i, e] = sum over the splits, in order, of partial[split][i][e]; four experts per thread,
// four partials in flight.
__global__ void route_dw_reduce_kernel(const float *__restrict__ partial, int splits, int d,
                                       int E, int NE, float *__restrict__ dw_router) {
  pdl_start();
  const int n4 = NE / 4;
  const size_t plane = size_t(d) * n4;
  const float4 *src = reinterpret_cast<const float4 *>(partial);
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < d * n4; idx += gridDim.x * blockDim.x) {
    const int i = idx / n4, e = 4 * (idx - i * n4);
    if (e >= E) continue;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int y = 0; y < splits; y += 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (y + u < splits) v[u] = src[(y + u) * plane + idx];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (y + u < splits) {
          acc[0] += v[u].x;
          acc[1] += v[u].y;
          acc[2] += v[u].z;
          acc[3] += v[u].w;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (e + c < E) dw_router[size_t(i) * E + e + c] = acc[c];
  }
}

__global__ void zero_f32_kernel(float *p, int n) {
  pdl_start();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0.f;
}

template <bool DW, int G, bool AHEAD = false>
int launch_route_mma(const char *name, dim3 grid, size_t smem, const CUtensorMap &a, const CUtensorMap &b,
                       const RouteTcParams &p, cudaStream_t s, const char *what) {
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(route_tc_kernel<DW, G, AHEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRtMaxSmem);
    if (e != cudaSuccess) return moe::cuda_status(e, what);
    attr_set = true;
  }
  MOE_LAUNCH(name, s, moe::launch_dep(route_tc_kernel<DW, G, AHEAD>, grid, kRtThreads, smem, s, a, b, p));
  return moe::launch_status(what);
}
// Tensor-core logits: splits W into its three bf16 terms (w3), then one CTA per
// (token tile, split). Returns the number of partial planes written in *splits.
int launch_route_tc(const uint16_t *x, const float *w, int T, int d, int E, int NE, uint16_t *w3,
                    float *partial, int32_t *counts, int *splits_out, cudaStream_t s) {
  const int NP = route_tc_np(E);
  const RtPlan plan = route_logits_plan(T, d, NP);
  const int MT = plan.MT, stages = plan.stages, splits = plan.splits;
  const size_t smem = route_tc_smem(NP, stages, MT);
  dim3 sgrid((d + 31) / 32, (NP + 31) / 32);
  MOE_LAUNCH("route_split_w", s, moe::launch_dep(route_split_w_kernel, sgrid, dim3(32, 8), 0, s, w, d, E, NP, w3, counts));
  if (int st = moe::launch_status("moe_route: split router weight")) return st;
  CUtensorMap mx, mw;
  int st;
  if ((st = moe::make_map(&mx, x, uint64_t(T), uint64_t(d), kRtBK, kRtBM, "router x"))) return st;
  if ((st = moe::make_map(&mw, w3, uint64_t(3 * NP), uint64_t(d), kRtBK, uint32_t(NP), "router w")))
    return st;
  RouteTcParams p;
  p.M = T;
  p.MT = MT;
  p.kb_per_split = plan.kb_per_split;
  p.nkb = (d + kRtBK - 1) / kRtBK;
  p.NP = NP;
  p.NE = NE;
  p.stages = stages;
  p.tmem_cols = route_tc_tmem_cols(NP, MT);
  p.partial = partial;
  dim3 grid((T + kRtBM * MT - 1) / (kRtBM * MT), splits);
  *splits_out = splits;
  // A two-stage ring holds too little to cover an HBM load's way (~1.1 us a k-block), so the x tile
  // of a stage's next use goes to L2 while this one loads: 78.0 / 72.6 us at T=32768, d=4096,
  // 128 experts, 62.2 / 56.3 at 64, 428 / 412 at T=65536, d=7168, 208. Not with more stages (no gain
  // at 28 and 112 experts, 3 stages), nor above 208 experts, where the weights are most of a stage
  // (277 / 283 at T=65536, d=4096, 240), nor where a tile's rows straddle 128-byte lines (36.6 / 45.9
  // at T=16545, d=3336, 49 experts; 30.7 / 32.8 at d=3360), nor over few k-blocks. Further ahead is
  // slower (73.4 us three, 79 eight k-blocks on), and so it is for x^T dZ (40.9 / 47.8 at T=35700,
  // d=2856, 57 experts).
  const bool ahead = stages == 2 && NP <= 208 && plan.kb_per_split >= 16 && d % 64 == 0 &&
                     (reinterpret_cast<uintptr_t>(x) & 127) == 0;
  const char *what = "moe_route: logits";
  return ahead ? launch_route_mma<false, 1, true>("route_logits", grid, smem, mx, mw, p, s, what)
               : launch_route_mma<false, 1, false>("route_logits", grid, smem, mx, mw, p, s, what);
}

int launch_route(const uint16_t *x, const float *w, const float *b, const uint8_t *mask, int T,
                 int d, int E, int k, const float *lin, float *lout, int32_t *idx, float *gate,
                 int32_t *counts, float *partial, uint16_t *w3, cudaStream_t s) {
  int splits = 0;
  const int NE = padded_experts(E);
  if (lin == nullptr)
    if (int st = launch_route_tc(x, w, T, d, E, NE, w3, partial, counts, &splits, s)) return st;
  // at most eight blocks per SM, so that each block's shared histogram sums ~50 tokens'
  // assignments or more before its global atomics (one block per 8 tokens sent 512k atomics to
  // the counters at T=65536, top-8; the heaviest expert's counter took ~60k of them one after
  // another)
  const bool wide = T <= 2048;  // 16 lanes per token: 6.5 against 16 us at T=764, 198 experts, 13 against 7 at T=8192, 64
  const int per_block = kTopkThreads / (wide ? 16 : 4);
  const int grid = int(std::min<int64_t>((int64_t(T) + per_block - 1) / per_block, int64_t(moe::num_sms()) * 8));
  auto launch = [&](auto kern) {
    MOE_LAUNCH("route_topk", s, moe::launch_dep(kern, grid, kTopkThreads, 0, s, partial, splits, NE, lin, b, mask, T, E,
                                                k, lout, idx, gate, counts));
  };
  if (k <= 2) launch(wide ? route_topk_kernel<2, 16> : route_topk_kernel<2, 4>);
  else if (k <= 4) launch(wide ? route_topk_kernel<4, 16> : route_topk_kernel<4, 4>);
  else launch(wide ? route_topk_kernel<8, 16> : route_topk_kernel<8, 4>);
  return moe::launch_status("moe_route: top-k");
}

}  // namespace

namespace moe {
MOE_DEV_ERR_DEFINE_READER(route_dev_error)

size_t route_partial_bytes(int T, int d, int E) {
  if (T <= 0) return 0;
  const int splits = route_logits_plan(T, d, route_tc_np(E)).splits;
  return size_t(splits) * size_t(T) * size_t(padded_experts(E)) * 4;
}
size_t route_w3_bytes(int d, int E) { return size_t(3) * route_tc_np(E) * size_t(d) * 2; }
size_t route_dz3_bytes(int T, int E) {
  return size_t(3) * route_tc_np(E) * size_t(route_tokens_padded(T)) * 2;
}
size_t route_dw_partial_bytes(int T, int d, int E) {
  if (T <= 0) return 0;
  const int splits = route_dw_plan(d, route_tokens_padded(T), route_tc_np(E)).splits;
  return size_t(splits) * size_t(d) * size_t(route_dw_stride(E)) * 4;
}
}  // namespace moe

extern "C" {

int moe_route(const uint16_t *x, const float *w_router, const float *bias,
              const uint8_t *active_mask, int T, int d, int E, int k, const float *logits_in,
              float *logits_out, int32_t *topk_idx, float *topk_gate, int32_t *counts, void *ws,
              size_t ws_bytes, moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256) return moe::set_error(MOE_ERR_UNSUPPORTED, "moe_route: E=%d not in [1,256]", E);
  if (k < 1 || k > 8 || k > E) return moe::set_error(MOE_ERR_UNSUPPORTED, "moe_route: k=%d", k);
  if (T < 0 || d <= 0 || d % 8) return moe::set_error(MOE_ERR_ARG, "moe_route: T=%d d=%d", T, d);
  if (T > 0 && (!topk_idx || !topk_gate)) return moe::set_error(MOE_ERR_ARG, "moe_route: null output");
  if (T > 0 && !logits_in && (!x || !w_router))
    return moe::set_error(MOE_ERR_ARG, "moe_route: null x/w_router");
  if (x && !moe::aligned16(x)) return moe::set_error(MOE_ERR_ARG, "moe_route: x not 16-byte aligned");
  float *partial = nullptr;
  uint16_t *w3 = nullptr;
  if (!logits_in && T > 0) {
    const moe::WsLayout L = moe::ws_layout(T, d, E, k, 0);
    if (!ws || ws_bytes < L.total) return moe::set_error(MOE_ERR_WORKSPACE, "moe_route: workspace");
    if (!moe::aligned16(ws)) return moe::set_error(MOE_ERR_ARG, "moe_route: ws alignment");
    partial = reinterpret_cast<float *>(static_cast<char *>(ws) + L.route_partial);
    w3 = reinterpret_cast<uint16_t *>(static_cast<char *>(ws) + L.route_w3);
  }
  if (counts && (logits_in || T == 0)) {  // else zeroed by the kernel that splits w_router
    MOE_LAUNCH("zero_counts", s, moe::launch_dep(zero_i32_kernel, 1, 256, 0, s, counts, E));
    if (int st = moe::launch_status("moe_route: zero counts")) return st;
  }
  if (T == 0) return MOE_OK;
  return launch_route(x, w_router, bias, active_mask, T, d, E, k, logits_in, logits_out, topk_idx, topk_gate, counts,
                      partial, w3, s);
}

int moe_load_stats(const int32_t *topk_idx, int T, int k, int E, int32_t *counts, int accumulate,
                   moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || T < 0) return moe::set_error(MOE_ERR_ARG, "moe_load_stats: sizes");
  if (!counts || (T > 0 && !topk_idx)) return moe::set_error(MOE_ERR_ARG, "moe_load_stats: null");
  const int64_t A = int64_t(T) * k;
  if (!accumulate && A <= 8192) {  // one block (8 loads per thread), no launch to zero the counts
    MOE_LAUNCH("load_stats", s, moe::launch_dep(load_stats_kernel, 1, 1024, 0, s, topk_idx, A, E, 1, counts));
    return moe::launch_status("moe_load_stats: launch");
  }
  if (!accumulate) {
    MOE_LAUNCH("zero_counts", s, moe::launch_dep(zero_i32_kernel, 1, 256, 0, s, counts, E));
    if (int st = moe::launch_status("moe_load_stats: zero")) return st;
  }
  if (A == 0) return MOE_OK;
  const int grid = int(std::min<int64_t>((A + 255) / 256, int64_t(moe::num_sms()) * 4));
  MOE_LAUNCH("load_stats", s, moe::launch_dep(load_stats_kernel, grid, 256, 0, s, topk_idx, A, E, 0, counts));
  return moe::launch_status("moe_load_stats: launch");
}

}  // extern "C"

namespace {
// Weight-gradient launch on the tensor cores: partial[split][i][e] over the split's tokens.
int launch_route_dw(const uint16_t *x, const uint16_t *dz3, int T, int d, int E, float *partial,
                    int *splits_out, cudaStream_t s) {
  const int NP = route_tc_np(E), Tp = route_tokens_padded(T);
  const RtPlan plan = route_dw_plan(d, Tp, NP);
  const int MT = plan.MT, stages = plan.stages, splits = plan.splits;
  const size_t smem = route_tc_smem(NP, stages, MT);
  CUtensorMap mx, mz;
  int st;
  // x [T, d] read as 64 features x 64 tokens boxes (features contiguous: MN-major A)
  if ((st = moe::make_map(&mx, x, uint64_t(T), uint64_t(d), 64, kRtBK, "router bwd x"))) return st;
  if ((st = moe::make_map(&mz, dz3, uint64_t(3 * NP), uint64_t(Tp), kRtBK, uint32_t(NP), "router bwd dz")))
    return st;
  RouteTcParams p;
  p.M = d;
  p.MT = MT;
  p.kb_per_split = plan.kb_per_split;
  p.nkb = Tp / kRtBK;
  p.NP = NP;
  p.NE = route_dw_stride(E);
  p.stages = stages;
  p.tmem_cols = route_tc_tmem_cols(route_dw_group(NP) * NP, MT);
  p.partial = partial;
  dim3 grid((d + kRtBM * MT - 1) / (kRtBM * MT), splits);
  *splits_out = splits;
  const char *what = "moe_route_bwd: weight gradient";
  switch (route_dw_group(NP)) {
    case 1: return launch_route_mma<true, 1>("route_bwd_dw", grid, smem, mx, mz, p, s, what);
    case 2: return launch_route_mma<true, 2>("route_bwd_dw", grid, smem, mx, mz, p, s, what);
    default: return launch_route_mma<true, 3>("route_bwd_dw", grid, smem, mx, mz, p, s, what);
  }
}
}  // namespace

extern "C" {

int moe_route_bwd(const uint16_t *x, const int32_t *topk_idx, const float *topk_gate,
                  const float *d_gate, int T, int d, int E, int k, float *d_logits,
                  float *dw_router, void *ws, size_t ws_bytes, moe_stream_t stream) {
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (E < 1 || E > 256 || k < 1 || k > 8 || k > E || T < 0 || d <= 0 || d % 8)
    return moe::set_error(MOE_ERR_ARG, "moe_route_bwd: sizes");
  if (!dw_router || (T > 0 && (!x || !topk_idx || !topk_gate || !d_gate || !d_logits || !ws)))
    return moe::set_error(MOE_ERR_ARG, "moe_route_bwd: null pointer");
  if ((x && !moe::aligned16(x)) || (ws && !moe::aligned16(ws)))
    return moe::set_error(MOE_ERR_ARG, "moe_route_bwd: alignment");
  if (T == 0) {
    const int n = d * E;
    MOE_LAUNCH("zero_dw_router", s, moe::launch_dep(zero_f32_kernel, std::min((n + 255) / 256, 1024), 256, 0, s, dw_router, n));
    return moe::launch_status("moe_route_bwd: zero");
  }
  const moe::WsLayout L = moe::ws_layout(T, d, E, k, 0);
  if (ws_bytes < L.total) return moe::set_error(MOE_ERR_WORKSPACE, "moe_route_bwd: workspace");
  uint16_t *dz3 = reinterpret_cast<uint16_t *>(static_cast<char *>(ws) + L.route_dz3);
  float *partial = reinterpret_cast<float *>(static_cast<char *>(ws) + L.route_dw_partial);
  const int NP = route_tc_np(E), Tp = route_tokens_padded(T);
  dim3 zgrid((Tp + 255) / 256, (NP + kDzExperts - 1) / kDzExperts);
  MOE_LAUNCH("route_bwd_dz", s, moe::launch_dep(route_bwd_dz_kernel, zgrid, 256, 0, s,
                                    topk_idx, topk_gate, d_gate, T, Tp, k, NP, d_logits, dz3));
  if (int st = moe::launch_status("moe_route_bwd: dz")) return st;
  int splits = 0;
  if (int st = launch_route_dw(x, dz3, T, d, E, partial, &splits, s)) return st;
  const int n = d * (route_dw_stride(E) / 4);
  MOE_LAUNCH("route_bwd_reduce", s, moe::launch_dep(route_dw_reduce_kernel, std::min((n + 255) / 256, 4 * moe::num_sms()), 256, 0, s,
                                        partial, splits, d, E, route_dw_stride(E), dw_router));
  return moe::launch_status("moe_route_bwd: reduce");
}

}  // extern "C"
