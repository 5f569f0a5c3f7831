// Backward pass of the UniF-MoE layer (training, Sec. III-E) for bf16 layers,
// on the tensor cores, over the group table of the forward that preceded it.
//
// The discrete decisions (b, I_shr, k and the selected experts) are
// piecewise constant in the parameters, so gradients flow through the
// pathway weights alpha (Eq. 18) and s_j (Eq. 24) and through the experts
// (Eq. 16). For a group row (token t, expert e, block b) with weight w and
// pre-activations a = x K_e[:, H_b]:
//   g      = dy V_e[H_b, :]^T                 (the output gradient per channel)
//   dL/da  = w g GeLU'(a)                     -> DA row
//   w GeLU(a)                                 -> HW row
//   dL/dw += sum_h GeLU(a_h) g_h              -> dwt[t][e] (alpha for e = 0, s_j for e = 1+j)
// then, summed over rows:
//   dL/dx[t]          += DA row K_e[H_b, :]   (the streaming down kernel on K^T)
//   dL/dK_e[H_b, :]    = DA^T X[rows]         (weight-gradient kernel)
//   dL/dV_e[:, H_b]    = DY[rows]^T HW        (same kernel)
// and per token dL/dz from dL/dalpha and dL/ds (Eqs. 18, 24), dL/dW* = X^T dL/dz,
// dL/dbias = sum dL/dz, dL/dx += dL/dz W*^T; the Gram regulariser (Eq.
// diversity-loss) adds lambda_div dL_div/dW*.
//
// Kernels (in stream order): tile list from the forward's group sizes,
// bwd_hidden_kernel (CTA pairs, two tcgen05 accumulators: x K and dy V^T over
// the same gathered rows), the down kernel for dL/dx, bwd_wgrad_kernel (tcgen05 with
// MN-major operands: the token rows are the reduction dimension), the
// router-gradient kernels and the Gram kernel. Every wait on an mbarrier is
// bounded; a wait that runs out records kStatusTimeout and the CTA unwinds.
#include <stdio.h>

#include <algorithm>

#include "decide.cuh"
#include "internal.cuh"
#include "tc_common.cuh"

namespace unif {
namespace tc {
namespace bwd {

// GeLU (exact erf form, Sec. II-A) and its derivative Phi(a) + a phi(a).
// GeLU's value goes into dL/dalpha and dL/ds in fp32, so Phi is as exact as
// erff would make it. The hidden kernel's epilogue is bound by these
// instructions, though, and the exponential that phi needs serves Phi as well:
//   |a| < 1.35: Phi(a) = 1/2 + a P(a^2), P of degree 5;
//   beyond:     Phi(-|a|) = exp(-a^2 / 2) t R(t), t = 1 / (1 + |a| / 2), R of degree 3
// (minimax fits, each coefficient rounded to fp32 before the next is fitted:
// tests/gelu_fit.py). Measured over [-8, 8]: Phi within 6.04e-8, rms 1.11e-8;
// 0.5 (1 + erff(a / sqrt 2)) within 6.73e-8, rms 1.58e-8, and no better in any of 14
// intervals. ViT-S, 12,608 tokens: 118 us, with erff 138. (One expression for all a,
// the erfc approximation 7.1.26 of Abramowitz and Stegun, took 111, but was within
// 3.4e-7 only.)
__device__ __forceinline__ void gelu_and_grad(float a, float& g, float& dg) {
  const float u = a * a;
  float e, t;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(u * -0.72134752044448170f));  // exp(-a^2/2)
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(fabsf(a), 0.5f, 1.0f)));
  float p = fmaf(-6.28209773e-06f, u, 0.00010880574f);  // P
  p = fmaf(p, u, -0.00118041399f);
  p = fmaf(p, u, 0.00997000933f);
  p = fmaf(p, u, -0.0664895996f);
  p = fmaf(p, u, 0.398942232f);
  float r = fmaf(-0.145465598f, t, 0.275724202f);  // R
  r = fmaf(r, t, 0.164777622f);
  r = fmaf(r, t, 0.203067407f);
  const float tail = fmaf(-copysignf(r * t, a), e, a > 0.f ? 1.f : 0.f);
  const float cdf = fabsf(a) < 1.35f ? fmaf(a, p, 0.5f) : tail;
  g = a * cdf;
  dg = fmaf(a * 0.39894228040143268f, e, cdf);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Instruction descriptor of kind::f16 (bf16 in, fp32 accumulate) with both
// operands MN-major (transpose bits 15 and 16).
__device__ __forceinline__ uint32_t idesc_bf16_mn(int m, int n) {
  return idesc_bf16(m, n) | (1u << 15) | (1u << 16);
}

// Shared-memory descriptor of an MN-major operand with the 128-byte swizzle:
// each 128-byte row holds 64 consecutive MN elements of one K index, 8-row
// (K) groups are 1024 bytes apart (stride-dimension offset), and blocks of
// 64 MN elements are `lbo` bytes apart (leading-dimension offset).
__device__ __forceinline__ uint64_t sw128_mn_desc(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

constexpr int kEpiWarps = 8;      // of the weight-gradient kernel
// Most 128-row tiles that one accumulation of the weight gradients runs over:
// the tensor cores truncate the accumulator at every 16 rows, so the error grows
// with the number of rows. Further rows are added in fp32.
constexpr int kSumTiles = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAcc2 = 256;   // TMEM column of the second accumulator

// Most 128-row tiles of a group in one weight-gradient item, `total` tiles in
// `parts` items each (features x channels x kinds) on `ctas` CTAs: as many as
// leave every CTA two items, so that most groups are one chunk, whose sums
// are stored instead of added into zeroed outputs. (ViT-S, 25 tiles per
// group: chunks of at most 8 took 101 us, this 95; BERT-base, 5
// tiles: 115 and 97, its 170 MB of gradients being more than L2 holds
// between the clearing and the adds.)
__device__ __forceinline__ int chunk_tiles(int total, int parts, int ctas) {
  return max(kSumTiles, (int)(((long long)total * parts + 2 * ctas - 1) / (2 * ctas)));
}

// ---------------------------------------------------------------------------
// bwd_hidden_kernel: per 256-row tile of a group and N sub-tile, on a pair of
// CTAs (tcgen05 cta_group::2, M = 256, 128 rows each), acc_a = X[rows]
// K_e[cols]^T and acc_g = DY[rows] V_e^T[cols]^T (both reductions over d),
// then the epilogue of the header comment.
// Roles (each CTA, 18 warps): warps 0-7 gather this CTA's 128 rows of a
// step, a warp per ring stage (even steps x rows, odd steps dy rows: each
// 64-deep k-block takes one of each); warp 8 brings this CTA's half of the
// step's weight tile (keys, values) by TMA; warp 9 allocates TMEM and, in
// the even CTA, issues the MMAs; warps 10-17 run the epilogue (warp w: TMEM
// lane quarter w % 4, one half of the columns), which leaves 32 x 32 pieces
// of both outputs in shared memory for TMA stores (64-byte swizzle). The two
// accumulators take 2 bn <= 512 TMEM columns, so a tile's MMAs wait for the
// epilogue of the one before; the ring holds the next tile's first steps by
// then. (16 epilogue warps of half the columns ran no faster.)
// Measured (one CTA per tile, four gather warps, erff, a 32-byte row piece per
// thread's store before): ViT-S (12,608 tokens) 138 -> 118 us; BERT-base (2,300
// tokens) 102 -> 77.
// ---------------------------------------------------------------------------
struct HiddenParams {
  const int32_t* counts;   // [G] group sizes (the forward's)
  int G, region;
  const int32_t* row_tok;  // [G][region]
  const float* row_w;
  const __nv_bfloat16* x;
  const __nv_bfloat16* dy;
  float* dwt;          // [T][K+1]
  // outputs that later kernels add into, zeroed here by the odd CTAs' MMA
  // warps (which have no MMAs to issue): dw_up and dw_down of the experts with
  // a group that is no single weight-gradient chunk (w_parts items per chunk
  // on w_ctas CTAs), dw_router (n_wr floats), dbias (n_bias floats)
  float* dw_up;
  float* dw_down;
  float* dw_router;
  float* dbias;
  int w_parts, w_ctas;
  int n_wr, n_bias;
  int n_sub, bn, num_kb, B, M, H, d, K1, stages;
  int* status;
  long long wait_limit;
};

constexpr int kHGather = 8;     // at most one warp per ring stage
constexpr int kHLoader = 8, kHMma = 9, kHFirstEpi = 10, kHEpiWarps = 8;
constexpr int kHThreads = 32 * (kHFirstEpi + kHEpiWarps);  // 576
constexpr int kHMinStages = 4;
constexpr int kHPairRows = 256;
constexpr uint32_t kHPiece = 32u * 64u;  // 32 rows x 32 bf16
constexpr uint32_t kHStaging = kHEpiWarps * 2u * kHPiece;
constexpr uint32_t kHBarBytes = 256;
constexpr uint32_t kHZero = 4096;  // zeros, the source of the bulk stores that clear the outputs

__host__ __device__ constexpr uint32_t hidden_stage_bytes(int bn) {
  return kStageA + (uint32_t)bn * 64u;
}
__host__ __device__ constexpr uint32_t hidden_smem_bytes(int bn, int stages, int G) {
  return 1024u + (uint32_t)stages * hidden_stage_bytes(bn) + kHStaging + kHZero + kHBarBytes +
         (uint32_t)((3 * G + 2) * 4 + 15) / 16u * 16u;
}

// A bounded wait that ignores the abort flag (copies and MMAs in flight land
// before the pair releases its TMEM).
__device__ __forceinline__ void wait_settle(uint32_t bar, uint32_t parity, long long limit) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > limit) return;
}

__global__ void __launch_bounds__(kHThreads, 1)
bwd_hidden_kernel(const __grid_constant__ CUtensorMap tm_wk, const __grid_constant__ CUtensorMap tm_wv,
                  const __grid_constant__ CUtensorMap tm_da, const __grid_constant__ CUtensorMap tm_hw,
                  HiddenParams p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned base, the same offset in both CTAs of the pair
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int n_st = p.stages;
  const uint32_t stage_bytes = hidden_stage_bytes(p.bn);
  const uint32_t s0 = smem_u32(smem);
  // stage s: [128 rows x 64][bn / 2 weight rows x 64]
  auto sa = [&](int s) { return s0 + (uint32_t)s * stage_bytes; };
  auto sw = [&](int s) { return s0 + (uint32_t)s * stage_bytes + kStageA; };
  uint8_t* staging = smem + (size_t)n_st * stage_bytes;
  uint8_t* zeros = staging + kHStaging;
  uint64_t* bars = reinterpret_cast<uint64_t*>(zeros + kHZero);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kHGather + s); };
  const uint32_t accf = bar0 + 8u * (2 * kHGather);
  const uint32_t acce = bar0 + 8u * (2 * kHGather + 1);
  const uint32_t mma_done = bar0 + 8u * (2 * kHGather + 2);
  const uint32_t fin = bar0 + 8u * (2 * kHGather + 3);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kHGather + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert(8 * (2 * kHGather + 5) <= kHBarBytes, "barrier region");
  // first 256-row pair tile and first 128-row tile of every group, its size
  int32_t* first_s = reinterpret_cast<int32_t*>(reinterpret_cast<uint8_t*>(bars) + kHBarBytes);
  int32_t* first128_s = first_s + p.G + 1;
  int32_t* cnt_s = first128_s + p.G + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  auto arrive_leader = [&](uint32_t bar) {
    if (leader) mbar_arrive(bar);
    else mbar_arrive_cluster(mapa_shared(bar, 0));
  };
  if (threadIdx.x == 0) {
    for (int s = 0; s < kHGather; ++s) {
      mbar_init(full_bar(s), 3);  // an owner warp of each CTA, the leader's loader
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, 2 * kHEpiWarps);
    mbar_init(mma_done, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kHMma) {
    tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish_pair();
  }
  for (int g = threadIdx.x; g < p.G; g += kHThreads) cnt_s[g] = min(p.counts[g], p.region);
  __syncthreads();
  if (warp == 0) {
    tile_scan<kBM>(p.G, lane, first128_s, cnt_s);
  } else if (warp == 1) {
    tile_scan<kHPairRows>(p.G, lane, first_s, cnt_s);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers are initialised before either CTA signals the other
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int n_items = first_s[p.G] * p.n_sub;
  // group, sub-tile, this CTA's first row in the group and its real rows
  struct Item { int g, ns, pos, rows; };
  auto item_of = [&](int item) {
    Item it;
    const int tile = item / p.n_sub;
    it.ns = item - tile * p.n_sub;
    int lo = 0, hi = p.G - 1;  // the last group whose first pair tile is <= tile
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first_s[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    it.g = lo;
    it.pos = kHPairRows * (tile - first_s[lo]) + kBM * (int)rank;
    it.rows = max(0, min(kBM, cnt_s[lo] - it.pos));
    return it;
  };
  const int n_steps = 2 * p.num_kb;  // step 2 kb: x and keys, 2 kb + 1: dy and values

  if (warp < kHGather) {
    // ---- this CTA's rows of the steps of stage `warp` ----
    const int j = lane & 7, rsub = lane >> 3;
    const uint32_t dst = sa(warp);
    bool ok = true;
    uint32_t ph = 0;
    int ks = warp;  // this warp's next step, counted from the item's first
    for (int item = pair; item < n_items && ok && warp < n_st; item += n_pairs) {
      if (ks < n_steps) {
        const Item it = item_of(item);
        int tk[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          tk[i] = 32 * i + lane < it.rows
                      ? p.row_tok[(size_t)it.g * p.region + it.pos + 32 * i + lane] : -1;
        for (; ks < n_steps; ks += n_st) {
          ok = wait_warp(empty_bar(warp), ph ^ 1u, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          ph ^= 1u;
          const __nv_bfloat16* sj = ((ks & 1) ? p.dy : p.x) + j * 8 + (ks >> 1) * kBK;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int r = 4 * i + rsub;
            const int t = __shfl_sync(0xffffffffu, tk[i >> 3], r & 31);
            // (padding rows keep what the stage holds: their results are dropped)
            if (t >= 0)
              cp_async16(dst + r * 128u + ((j ^ (r & 7)) << 4), sj + (size_t)t * p.d);
          }
          cp_async_commit();
          cp_async_wait<0>();
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) arrive_leader(full_bar(warp));
        }
      }
      ks -= n_steps;
    }
  } else if (warp == kHLoader) {
    // ---- this CTA's half of every step's weight tile ----
    bool ok = true;
    int s = 0;
    uint32_t ph = 0;
    long long issued = 0;
    for (int item = pair; item < n_items && ok; item += n_pairs) {
      const Item it = item_of(item);
      const int e = it.g / p.B, blk = it.g - e * p.B;
      const int row = e * p.H + blk * p.M + it.ns * p.bn + (int)rank * (p.bn / 2);
      for (int ks = 0; ks < n_steps; ++ks) {
        ok = wait_warp(empty_bar(s), ph ^ 1u, abort_flag, p.status, p.wait_limit);
        if (!ok) break;
        if (lane == 0) {
          if (leader) mbar_expect_tx(full_bar(s), (uint32_t)p.bn * 128u);
          tma_load_2d_pair(sw(s), (ks & 1) ? &tm_wv : &tm_wk, mapa_shared(full_bar(s), 0),
                           (ks >> 1) * kBK, row);
        }
        __syncwarp();
        ++issued;
        if (++s == n_st) { s = 0; ph ^= 1u; }
      }
    }
    // loads still in flight land before the pair exits
    if (leader && lane == 0)
      for (long long q = issued > n_st ? issued - n_st : 0; q < issued; ++q)
        wait_settle(full_bar((int)(q % n_st)), (uint32_t)((q / n_st) & 1), p.wait_limit / 16);
    __syncwarp();
  } else if (warp == kHMma) {
    // ---- MMA issuer (the leader CTA) ----
    if (leader) {
      const uint32_t idesc = idesc_bf16(2 * kBM, p.bn);
      const uint16_t both = 3;
      int s = 0;
      uint32_t ph = 0, acc_ph = 0;
      bool ok = true, any = false;
      for (int item = pair; item < n_items && ok; item += n_pairs) {
        ok = wait_warp_cluster(acce, acc_ph ^ 1u, abort_flag, p.status, p.wait_limit);
        if (!ok) break;
        tc_fence_after();
        for (int ks = 0; ks < n_steps; ++ks) {
          ok = wait_warp_cluster(full_bar(s), ph, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          tc_fence_after();
          // even steps feed x K (acc_a), odd ones dy V^T (acc_g)
          const uint32_t d_tmem = tmem_base + ((ks & 1) ? kAcc2 : 0u);
          if (elect_one()) {
            const uint64_t a = sw128_desc(sa(s)), b = sw128_desc(sw(s));
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16_pair(d_tmem, a + 2 * k, b + 2 * k, idesc, ((ks >> 1) | k) != 0 ? 1u : 0u);
            umma_commit_pair(empty_bar(s), both);
            if (ks == n_steps - 1) umma_commit_pair(accf, both);
          }
          __syncwarp();
          any = true;
          if (++s == n_st) { s = 0; ph ^= 1u; }
        }
        acc_ph ^= 1u;
      }
      // every MMA issued has completed before the pair releases TMEM
      if (any) {
        if (elect_one()) umma_commit_pair(mma_done, 1);
        __syncwarp();
        wait_settle(mma_done, 0u, p.wait_limit);
      }
    } else {
      for (uint32_t k = lane; k < kHZero / 16; k += 32)
        reinterpret_cast<uint4*>(zeros)[k] = make_uint4(0u, 0u, 0u, 0u);
      fence_proxy_async();
      __syncwarp();
      const int most = chunk_tiles(first128_s[p.G], p.w_parts, p.w_ctas);
      const long long bytes = (long long)p.H * p.d * 4;  // of one expert's dK or dV
      for (int e = 0; e < p.G / p.B; ++e) {
        // an expert with a block whose group is empty or split is cleared
        // whole (its other blocks are overwritten): its dV rows interleave
        // the blocks, and clearing them block by block took 50 us more
        bool clear = false;
        for (int blk = lane; blk < p.B; blk += 32) {
          const int nt = first128_s[e * p.B + blk + 1] - first128_s[e * p.B + blk];
          clear |= nt == 0 || nt > most;
        }
        if (!__any_sync(0xffffffffu, clear)) continue;
        uint8_t* up = reinterpret_cast<uint8_t*>(p.dw_up) + e * bytes;
        uint8_t* dn = reinterpret_cast<uint8_t*>(p.dw_down) + e * bytes;
        for (long long k = (long long)kHZero * (32 * pair + lane); k < bytes;
             k += (long long)kHZero * 32 * n_pairs) {
          const uint32_t n = (uint32_t)min((long long)kHZero, bytes - k);
          bulk_store(up + k, smem_u32(zeros), n);
          bulk_store(dn + k, smem_u32(zeros), n);
        }
      }
      bulk_commit();
      for (int k = 32 * pair + lane; k < p.n_wr; k += 32 * n_pairs) p.dw_router[k] = 0.f;
      for (int k = 32 * pair + lane; k < p.n_bias; k += 32 * n_pairs) p.dbias[k] = 0.f;
      bulk_wait_all();
    }
    __syncwarp();
  } else {
    // ---- epilogue ----
    const int q = warp & 3;
    const int cols = p.bn / 2, c_begin = ((warp - kHFirstEpi) >> 2) * cols;
    uint8_t* stg = staging + (size_t)(warp - kHFirstEpi) * 2 * kHPiece;
    uint8_t* srow = stg + lane * 64;
    const uint32_t sx = (uint32_t)(lane >> 1) & 3u;  // 64-byte swizzle of this row's chunks
    uint32_t acc_ph = 0;
    for (int item = pair; item < n_items; item += n_pairs) {
      const Item it = item_of(item);
      const int e = it.g / p.B;
      const int r = q * 32 + lane;
      const bool real = r < it.rows;
      const size_t lr = (size_t)it.g * p.region + it.pos + r;
      const int tok = real ? p.row_tok[lr] : -1;
      // (padding rows have weight 0: their outputs are zeros, which the
      // weight-gradient kernel sums over; see the finite selects below)
      const float w = real ? p.row_w[lr] : 0.f;
      if (!wait_warp(accf, acc_ph, abort_flag, p.status, p.wait_limit)) break;
      tc_fence_after();
      if (it.rows > 0) {  // (a half past the group's end has no tile of its own)
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + c_begin;
        // rows and columns of the outputs' tile (maps of 32 x 32 boxes)
        const int row0 = first128_s[it.g] * kBM + it.pos + q * 32;
        const int col0 = it.ns * p.bn + c_begin;
        float dot0 = 0.f, dot1 = 0.f;
        for (int c = 0; c < cols; c += 32) {
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {  // (all 32 columns at once: registers spill)
            float a[16], gv[16];
            uint32_t od[8], oh[8];
            tmem_ld16(t_row + c + 16 * hh, a);
            tmem_ld16(t_row + kAcc2 + c + 16 * hh, gv);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              // a padding row's accumulators may hold anything
              const float a0 = real ? a[2 * i] : 0.f, a1 = real ? a[2 * i + 1] : 0.f;
              const float v0 = real ? gv[2 * i] : 0.f, v1 = real ? gv[2 * i + 1] : 0.f;
              float g0, g1, dg0, dg1;
              gelu_and_grad(a0, g0, dg0);
              gelu_and_grad(a1, g1, dg1);
              dot0 = fmaf(g0, v0, dot0);
              dot1 = fmaf(g1, v1, dot1);
              od[i] = pack_bf16(w * v0 * dg0, w * v1 * dg1);
              oh[i] = pack_bf16(w * g0, w * g1);
            }
            if (hh == 0) {
              if (lane == 0) bulk_wait_read();  // the last pieces have left the staging
              __syncwarp();
            }
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
              const uint32_t ch = ((uint32_t)(2 * hh + jj) ^ sx) << 4;
              *reinterpret_cast<uint4*>(srow + ch) =
                  make_uint4(od[4 * jj], od[4 * jj + 1], od[4 * jj + 2], od[4 * jj + 3]);
              *reinterpret_cast<uint4*>(srow + kHPiece + ch) =
                  make_uint4(oh[4 * jj], oh[4 * jj + 1], oh[4 * jj + 2], oh[4 * jj + 3]);
            }
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&tm_da, smem_u32(stg), col0 + c, row0);
            tma_store_2d(&tm_hw, smem_u32(stg) + kHPiece, col0 + c, row0);
            bulk_commit();
          }
        }
        if (tok >= 0) atomicAdd(p.dwt + (size_t)tok * p.K1 + e, dot0 + dot1);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_leader(acce);
      acc_ph ^= 1u;
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
  }
  // every warp converged before the CTA barrier; then each CTA tells its peer
  // that it is done with the pair's TMEM (the leader after its MMAs
  // completed), and the owner warp waits for the peer's word
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) mbar_arrive_cluster(mapa_shared(fin, rank ^ 1u));
  if (warp == kHMma) {
    wait_settle(fin, 0u, p.wait_limit);
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// bwd_wgrad_kernel: per item (group g, a chunk of its rows, 128 features c of
// d, N chunk nc of the block's M channels, kind) one accumulator over the
// chunk's rows, 64 rows per stage:
//   kind 0: acc[i][h] = sum_r X[tok_r][c*128 + i] DA[r][nc*N + h]   -> dK_e (transposed)
//   kind 1: acc[i][h] = sum_r DY[tok_r][c*128 + i] HW[r][nc*N + h]  -> dV_e
// The token rows are the reduction dimension, so both operands are MN-major:
// the gathered rows (x, dy) and the TMA tiles (DA, HW) keep the 128-byte
// swizzled row layout, read with MN-major descriptors. A group's tiles are
// one chunk, whose sums are stored, or split evenly into chunks of at most
// chunk_tiles, whose partial sums are added into the (zeroed) outputs. A
// chunk's rows are summed in accumulations of at most kSumTiles tiles: the first
// stays in its TMEM accumulator, the others run in the second one and are added
// there by the epilogue warps in fp32. (Each added into the outputs instead:
// 122 us per ViT-S backward.) The next chunk begins in the second accumulator
// while the sum of this one goes out.
// Roles: warps 0-4 fill the ring, a warp per stage (the gathered rows, and
// the DA or HW tiles by TMA), warp 5 MMAs, warps 6-13 epilogue. The two
// kinds are items of their own so that one accumulator leaves room in TMEM
// for a second: an item's atomic adds run under the next one's MMAs. Bound
// by the operand bytes out of L2 (40 KB per 64 rows of 192 channels).
// Measured (both kinds in one item, accumulators not overlapped, four stages
// of 32 rows before): ViT-S 12,608 tokens 117 -> 95 us, BERT-base (2,300
// tokens) 130 -> 97.
// ---------------------------------------------------------------------------
struct WgradParams {
  const int32_t* counts;   // [G] group sizes (the forward's)
  const int32_t* row_tok;  // per-group regions of `region` rows
  const __nv_bfloat16* x;
  const __nv_bfloat16* dy;
  float* dw_up;    // [K+1][H][d]
  float* dw_down;  // [K+1][d][H]
  int G, region, B, M, H, d, N, n_nc, n_c, stages;
  int* status;
  long long wait_limit;
};

constexpr uint32_t kRows = 64;                 // group rows per stage
constexpr uint32_t kPBytes = 2u * kRows * 128u;  // 128 features x 64 rows (two 64-column blocks)
constexpr int kWStages = 5;                      // at most one stage per producer warp
constexpr int kWMinStages = 2;
constexpr int kWMma = 5, kWFirstEpi = 6;
constexpr int kWThreads = 32 * (kWFirstEpi + kEpiWarps);  // 448
constexpr int kParts = kBM / (int)kRows;         // stages per 128-row tile

__host__ __device__ constexpr uint32_t wgrad_stage_bytes(int N) {
  return kPBytes + (uint32_t)(N / 64) * kRows * 128u;
}
__host__ __device__ constexpr uint32_t wgrad_smem_bytes(int N, int stages, int G) {
  return 1024u + (uint32_t)stages * wgrad_stage_bytes(N) + 160u + 4u * (3u * (uint32_t)G + 2u) + 16u;
}

__global__ void __launch_bounds__(kWThreads, 1)
bwd_wgrad_kernel(const __grid_constant__ CUtensorMap tm_da, const __grid_constant__ CUtensorMap tm_hw,
                 WgradParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int n_st = p.stages;
  const uint32_t stage_bytes = wgrad_stage_bytes(p.N);
  const uint32_t qbytes = (uint32_t)(p.N / 64) * kRows * 128u;
  const uint32_t s0 = smem_u32(smem);
  // stage s: [x or dy rows][DA or HW tile]
  auto sp = [&](int s) { return s0 + (uint32_t)s * stage_bytes; };
  auto sq = [&](int s) { return s0 + (uint32_t)s * stage_bytes + kPBytes; };
  uint8_t* gen_base = smem;  // generic pointer for zero-filling padding rows
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)n_st * stage_bytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kWStages + s); };
  auto accf_bar = [&](int a) { return bar0 + 8u * (2 * kWStages + a); };
  auto acce_bar = [&](int a) { return bar0 + 8u * (2 * kWStages + 2 + a); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kWStages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert(8 * (2 * kWStages + 4) + 16 <= 160, "barrier region");
  int32_t* first_s = reinterpret_cast<int32_t*>(tmem_slot + 4);  // [G + 1] first tiles
  int32_t* cnt_s = first_s + p.G + 1;                             // [G] sizes
  int32_t* chunk_s = cnt_s + p.G;                                 // [G + 1] first chunks

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kWStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), kEpiWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kWMma) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  grid_dep_wait();  // dL/da, w GeLU(a), and the zeroed outputs
  if (warp == kWThreads / 32 - 1) {
    tile_table(p.counts, p.G, p.region, lane, first_s, cnt_s);
    __syncwarp();
    // the first chunk of every group (chunk_s[G] = all chunks)
    const int most = chunk_tiles(first_s[p.G], p.n_c * p.n_nc * 2, (int)gridDim.x);
    int carry = 0;
    for (int g0 = 0; g0 < p.G; g0 += 32) {
      const int g = g0 + lane;
      const int nch = g < p.G ? (first_s[g + 1] - first_s[g] + most - 1) / most : 0;
      int inc = nch;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      if (g < p.G) chunk_s[g] = carry + inc - nch;
      carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) chunk_s[p.G] = carry;
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int n_items = chunk_s[p.G] * p.n_c * p.n_nc * 2;
  // item -> (group g, its tiles [t0, t0 + nt) of one chunk, feature chunk c,
  // N chunk nc, kind); rows of the chunk start at row r0 of the group
  struct Item {
    int g, t0, nt, r0, c, nc, kind;
    bool whole;  // the group's only chunk
    __device__ __forceinline__ int sums() const { return (nt + kSumTiles - 1) / kSumTiles; }
    // tiles of its j-th accumulation
    __device__ __forceinline__ int tiles(int j) const {
      return nt * (j + 1) / sums() - nt * j / sums();
    }
  };
  auto decode = [&](int item) {
    Item it;
    it.kind = item & 1;
    int q = item >> 1;
    it.nc = q % p.n_nc;
    q /= p.n_nc;
    it.c = q % p.n_c;
    q /= p.n_c;
    int lo = 0, hi = p.G - 1;  // the last group whose first chunk is <= q
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (chunk_s[mid] <= q) lo = mid; else hi = mid - 1;
    }
    it.g = lo;
    const int k = q - chunk_s[lo], nch = chunk_s[lo + 1] - chunk_s[lo];
    const int tiles = first_s[lo + 1] - first_s[lo];
    const int ta = tiles * k / nch;
    it.t0 = first_s[lo] + ta;
    it.nt = tiles * (k + 1) / nch - ta;
    it.whole = nch == 1;
    it.r0 = ta * kBM;
    return it;
  };

  if (warp < kWStages) {
    // ---- producers: warp w owns stage w: the gathered rows, and lane 0
    // brings the DA or HW tile by TMA ----
    const int j = lane & 7, rsub = lane >> 3;
    bool ok = true;
    uint32_t ph = 0;
    int kt = warp;  // this warp's next stage, counted from the item's first
    for (int item = blockIdx.x; item < n_items && ok && warp < n_st; item += gridDim.x) {
      const Item it = decode(item);
      const int n_steps = it.nt * kParts;
      const int size = cnt_s[it.g];
      const CUtensorMap* tm = it.kind == 0 ? &tm_da : &tm_hw;
      const __nv_bfloat16* sj = (it.kind == 0 ? p.x : p.dy) + (size_t)it.c * 128 + j * 8;
      for (; kt < n_steps; kt += n_st) {
        ok = wait_warp(empty_bar(warp), ph ^ 1u, abort_flag, p.status, p.wait_limit);
        if (!ok) break;
        ph ^= 1u;
        if (lane == 0) {
          mbar_expect_tx_only(full_bar(warp), qbytes);
          const int crow = it.t0 * kBM + kt * (int)kRows;
          for (int b = 0; b < p.N / 64; ++b)
            tma_load_2d(sq(warp) + b * kRows * 128u, tm, full_bar(warp), it.nc * p.N + b * 64, crow);
        }
        // this step's row tokens: lane l holds rows l and 32 + l (-1: padding)
        int tk[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int rg = it.r0 + kt * (int)kRows + 32 * i + lane;
          tk[i] = rg < size ? p.row_tok[(size_t)it.g * p.region + rg] : -1;
        }
        const uint32_t dst = sp(warp);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
#pragma unroll
          for (int i = 0; i < (int)kRows / 4; ++i) {
            const int r = 4 * i + rsub;
            const int t = __shfl_sync(0xffffffffu, tk[i >> 3], r & 31);
            const uint32_t off = b * kRows * 128u + r * 128u + ((j ^ (r & 7)) << 4);
            if (t >= 0)
              cp_async16(dst + off, sj + (size_t)t * p.d + b * 64);
            else  // padding rows contribute zeros to the row sums
              *reinterpret_cast<uint4*>(gen_base + (dst - s0) + off) = make_uint4(0u, 0u, 0u, 0u);
          }
        }
        cp_async_commit();
        cp_async_wait<0>();
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar(warp));
      }
      kt -= n_steps;  // stages count on over the items
    }
  } else if (warp == kWMma) {
    const uint32_t idesc = idesc_bf16_mn(kBM, p.N);
    const uint32_t lbo = kRows * 128u;  // 64-element MN blocks of kRows rows
    int s = 0, first = 0;  // first: the accumulator of an item's first sum
    uint32_t ph = 0, acc_ph = 0;  // (a phase bit per accumulator)
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
      const Item it = decode(item);
      for (int j = 0; j < it.sums() && ok; ++j) {
        const int n_steps = it.tiles(j) * kParts;
        const int acc = j == 0 ? first : first ^ 1;
        ok = wait_warp(acce_bar(acc), ((acc_ph >> acc) & 1u) ^ 1u, abort_flag, p.status,
                       p.wait_limit);
        if (!ok) break;
        acc_ph ^= 1u << acc;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * kAcc2;
        for (int kt = 0; kt < n_steps; ++kt) {
          ok = wait_warp(full_bar(s), ph, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < (int)kRows / 16; ++k)  // 16 rows (two 8-row groups) per MMA
              umma_bf16(d_tmem, sw128_mn_desc(sp(s) + k * 2048u, lbo),
                        sw128_mn_desc(sq(s) + k * 2048u, lbo), idesc, (kt | k) != 0 ? 1u : 0u);
            umma_commit(empty_bar(s));
            if (kt == n_steps - 1) umma_commit(accf_bar(acc));
          }
          __syncwarp();
          if (++s == n_st) { s = 0; ph ^= 1u; }
        }
      }
      first ^= 1;
    }
  } else if (warp >= kWFirstEpi) {
    const int q = warp & 3;
    const int half = (warp - kWFirstEpi) >> 2;
    const int cols = p.N / 2;
    // (the caller's buffer need only be 16-byte aligned)
    const bool wide = (reinterpret_cast<uintptr_t>(p.dw_down) & 31u) == 0;
    int first = 0;
    uint32_t acc_ph = 0;
    auto wait_acc = [&](int acc) {
      const uint32_t phase = (acc_ph >> acc) & 1u;
      acc_ph ^= 1u << acc;
      const bool ok = wait_warp(accf_bar(acc), phase, abort_flag, p.status, p.wait_limit);
      tc_fence_after();
      return ok;
    };
    auto release = [&](int acc) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce_bar(acc));
    };
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
      const Item it = decode(item);
      const int e = it.g / p.B, blk = it.g % p.B;
      const int i = it.c * 128 + q * 32 + lane;  // this thread's feature
      const int h0 = blk * p.M + it.nc * p.N + half * cols;  // first channel of its columns
      const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + half * cols;
      const uint32_t t_sum = t_row + (uint32_t)first * kAcc2;
      ok = wait_acc(first);
      for (int j = 1; j < it.sums() && ok; ++j) {  // the first sum += the j-th
        ok = wait_acc(first ^ 1);
        if (!ok) break;
        const uint32_t t_part = t_row + (uint32_t)(first ^ 1) * kAcc2;
        for (int cc = 0; cc < cols; cc += 32) {
          uint32_t u[32], v[32];
          float sum[32];
          tmem_ld32_async(t_sum + cc, u);
          tmem_ld32_async(t_part + cc, v);
          tmem_wait_ld();
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) sum[jj] = __uint_as_float(u[jj]) + __uint_as_float(v[jj]);
          tmem_st32_async(t_sum + cc, sum);
        }
        tmem_wait_st();
        release(first ^ 1);
      }
      if (!ok) break;
      // a whole group's sums are stored; the chunks of a split one add theirs
      // (those outputs start at zero)
      if (it.kind == 0) {  // dK_e[h][i]: a warp's lanes are 32 features of one h
        float* col = p.dw_up + ((size_t)e * p.H + h0) * p.d + i;
        for (int cc = 0; cc < cols; cc += 32) {
          float v[32];
          tmem_ld32(t_sum + cc, v);
          if (it.whole) {
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) col[(size_t)(cc + jj) * p.d] = v[jj];
          } else {
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) atomicAdd(col + (size_t)(cc + jj) * p.d, v[jj]);
          }
        }
      } else {  // dV_e[i][h]: a thread's columns are contiguous
        float* row = p.dw_down + ((size_t)e * p.d + i) * p.H + h0;
        for (int cc = 0; cc < cols; cc += 32) {
          float v[32];
          tmem_ld32(t_sum + cc, v);
          if (it.whole && wide) {  // whole 32-byte sectors per lane
#pragma unroll
            for (int jj = 0; jj < 32; jj += 8)
              asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                               row + cc + jj),
                           "f"(v[jj]), "f"(v[jj + 1]), "f"(v[jj + 2]), "f"(v[jj + 3]),
                           "f"(v[jj + 4]), "f"(v[jj + 5]), "f"(v[jj + 6]), "f"(v[jj + 7])
                           : "memory");
          } else if (it.whole) {
#pragma unroll
            for (int jj = 0; jj < 32; jj += 4)
              *reinterpret_cast<float4*>(row + cc + jj) =
                  make_float4(v[jj], v[jj + 1], v[jj + 2], v[jj + 3]);
          } else {
#pragma unroll
            for (int jj = 0; jj < 32; jj += 4)
              atomicAdd(reinterpret_cast<float4*>(row + cc + jj),
                        make_float4(v[jj], v[jj + 1], v[jj + 2], v[jj + 3]));
          }
        }
      }
      release(first);
      first ^= 1;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == kWMma) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Router gradients (Eqs. 17, 18, 24)
// ---------------------------------------------------------------------------
// dL/dz of token t into z[0..KC) (K + 1 <= KC values, the rest and a padding
// token's all zero): dL/dz_0 = dL/dalpha (1 - 2 tau) sigma(z_0)(1 - sigma(z_0))
// (adaptive alpha; sigma(z_0) = (alpha - tau) / (1 - 2 tau) from the stored
// alpha), dL/dz_{1+j} = s_j (dL/ds_j - sum_l s_l dL/ds_l), from the pathway
// weights' gradients dL/dalpha, dL/ds_j that the hidden kernel accumulated.
// All of the token's loads go out before the arithmetic.
template <int KC>
__device__ __forceinline__ void router_token_dz(int t, int K, float tau, int adaptive,
                                                const uint8_t* __restrict__ mask,
                                                const float* __restrict__ alpha,
                                                const float* __restrict__ s,
                                                const float* __restrict__ dwt, float (&z)[KC]) {
  const int K1 = K + 1;
  const bool valid = !mask || mask[t];
  const float* st = s + (size_t)t * K;
  const float* gt = dwt + (size_t)t * K1;
  float sv[KC], gv[KC];
#pragma unroll
  for (int j = 0; j < KC; ++j) {
    sv[j] = valid && j < K ? st[j] : 0.f;
    gv[j] = valid && j < K1 ? gt[j] : 0.f;
  }
  const float al = valid ? alpha[t] : 0.f;
  float part = 0.f;
#pragma unroll
  for (int j = 0; j + 1 < KC; ++j) part += sv[j] * gv[1 + j];
  z[0] = 0.f;
  if (valid && adaptive && tau < 0.5f) {
    const float sg = (al - tau) / (1.0f - 2.0f * tau);
    z[0] = gv[0] * (1.0f - 2.0f * tau) * sg * (1.0f - sg);
  }
#pragma unroll
  for (int j = 0; j + 1 < KC; ++j) z[1 + j] = sv[j] * (gv[1 + j] - part);
}

// dL/dz of every token into dz [T][K+1] (a thread per token).
template <int KC>
__global__ void __launch_bounds__(256)
router_dz_kernel(int T, int K, float tau, int adaptive, const uint8_t* __restrict__ mask,
                 const float* __restrict__ alpha, const float* __restrict__ s,
                 const float* __restrict__ dwt, float* __restrict__ dz) {
  grid_dep_wait();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  float z[KC];
  router_token_dz<KC>(t, K, tau, adaptive, mask, alpha, s, dwt, z);
  float* o = dz + (size_t)t * (K + 1);
#pragma unroll
  for (int c = 0; c < KC; ++c)
    if (c <= K) o[c] = z[c];
}

// dx[t][8 f .. 8 f + 8) = sum_c dL/dz_c(t) W*^T[c][8 f .. 8 f + 8) for the
// two tokens t = 2 p, 2 p + 1: a thread per (token pair, 8 features), so that
// each W*^T load serves both tokens. W*^T is the router's first K+1 columns
// as fp32 [K+1][d]; d % 128 == 0; padding tokens have dL/dz = 0 and get 0.
// Runs before the experts' share is added, so that dx is neither zeroed
// first nor read here.
__global__ void __launch_bounds__(256)
router_dx_kernel(int T, int K1, int d, const float* __restrict__ dz,
                 const float* __restrict__ wrT, float* __restrict__ dx) {
  grid_dep_wait();
  const int per = d / 8;
  const int n = ((T + 1) / 2) * per;
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < n; it += gridDim.x * blockDim.x) {
    const int p = it / per, f8 = it - p * per;
    const int ta = 2 * p, tb = min(2 * p + 1, T - 1);  // (tb == ta: the last odd token)
    float4* pa = reinterpret_cast<float4*>(dx + (size_t)ta * d + 8 * f8);
    float4* pb = reinterpret_cast<float4*>(dx + (size_t)tb * d + 8 * f8);
    const float* za = dz + (size_t)ta * K1;
    const float* zb = dz + (size_t)tb * K1;
    float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0, b0 = a0, b1 = a0;
    // four columns at a time: their loads go out together
    for (int cb = 0; cb < K1; cb += 4) {
      float4 w0[4], w1[4];
      float u[4], v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = cb + k;
        if (c < K1) {
          const float4* wc = reinterpret_cast<const float4*>(wrT + (size_t)c * d + 8 * f8);
          w0[k] = wc[0];
          w1[k] = wc[1];
          u[k] = za[c];
          v[k] = zb[c];
        } else {
          w0[k] = w1[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          u[k] = v[k] = 0.f;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        a0.x = fmaf(u[k], w0[k].x, a0.x); a0.y = fmaf(u[k], w0[k].y, a0.y);
        a0.z = fmaf(u[k], w0[k].z, a0.z); a0.w = fmaf(u[k], w0[k].w, a0.w);
        a1.x = fmaf(u[k], w1[k].x, a1.x); a1.y = fmaf(u[k], w1[k].y, a1.y);
        a1.z = fmaf(u[k], w1[k].z, a1.z); a1.w = fmaf(u[k], w1[k].w, a1.w);
        b0.x = fmaf(v[k], w0[k].x, b0.x); b0.y = fmaf(v[k], w0[k].y, b0.y);
        b0.z = fmaf(v[k], w0[k].z, b0.z); b0.w = fmaf(v[k], w0[k].w, b0.w);
        b1.x = fmaf(v[k], w1[k].x, b1.x); b1.y = fmaf(v[k], w1[k].y, b1.y);
        b1.z = fmaf(v[k], w1[k].z, b1.z); b1.w = fmaf(v[k], w1[k].w, b1.w);
      }
    }
    pa[0] = a0;
    pa[1] = a1;
    if (tb != ta) {
      pb[0] = b0;
      pb[1] = b1;
    }
  }
}

// dL/dW*[i][c] = sum_t x[t][i] dL/dz_c(t) and dL/dbias[c] = sum_t dL/dz_c(t):
// block (fc, j, cc) takes features [128 fc, 128 fc + 128), the tokens of
// slice j (kRwSlice tokens) and columns [16 cc, 16 cc + 16); 32 tokens at a
// time, the tile of x (16-byte loads; zero rows for padding tokens, whose x
// may hold anything) and of dL/dz go to shared memory (the next tile's
// loads run while the current tile is summed), then thread (g, q)
// adds x[t][2 q .. 2 q + 2) times dL/dz_{16 cc + 4 g .. + 4}(t) into its
// 2 x 4 partial sums (one 4-byte and one 16-byte shared load per 8 FMAs),
// which go out with one atomic add each.
constexpr int kRwSlice = 128;
__global__ void __launch_bounds__(256)
router_dw_kernel(int T, int K1, int d, const uint8_t* __restrict__ mask,
                 const __nv_bfloat16* __restrict__ x, const float* __restrict__ dz,
                 float* __restrict__ dw_router, float* __restrict__ dbias) {
  __shared__ __align__(16) __nv_bfloat16 xs[32][128];
  __shared__ __align__(16) float zs[32][16];
  grid_dep_wait();
  const int i0 = blockIdx.x * 128, c0 = blockIdx.z * 16;
  const int t_begin = blockIdx.y * kRwSlice, t_end = min(T, t_begin + kRwSlice);
  const int q = threadIdx.x & 63, g = threadIdx.x >> 6;
  const int lq = threadIdx.x & 15, lr = threadIdx.x >> 4;
  float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  float bacc[4] = {0.f, 0.f, 0.f, 0.f};
  // this thread's share of a tile: 16-byte chunk lq of x rows lr, lr + 16
  // and column c0 + lq of dL/dz for the same two tokens; the next tile's
  // share is loaded into registers while the current one is summed
  uint4 xr[2];
  float zr[2];
  auto load = [&](int tt) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int t = tt + lr + 16 * k, c = c0 + lq;
      xr[k] = make_uint4(0u, 0u, 0u, 0u);
      if (t < t_end && (!mask || mask[t]))
        xr[k] = reinterpret_cast<const uint4*>(x + (size_t)t * d + i0)[lq];
      zr[k] = t < t_end && c < K1 ? dz[(size_t)t * K1 + c] : 0.f;
    }
  };
  load(t_begin);
  for (int tt = t_begin; tt < t_end; tt += 32) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      reinterpret_cast<uint4*>(&xs[lr + 16 * k][0])[lq] = xr[k];
      zs[lr + 16 * k][lq] = zr[k];
    }
    __syncthreads();
    if (tt + 32 < t_end) load(tt + 32);
    const int nr = min(32, t_end - tt);
    for (int r = 0; r < nr; ++r) {
      const float2 xv = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&xs[r][0])[q]);
      const float4 z = reinterpret_cast<const float4*>(&zs[r][0])[g];
      acc[0][0] = fmaf(xv.x, z.x, acc[0][0]); acc[0][1] = fmaf(xv.x, z.y, acc[0][1]);
      acc[0][2] = fmaf(xv.x, z.z, acc[0][2]); acc[0][3] = fmaf(xv.x, z.w, acc[0][3]);
      acc[1][0] = fmaf(xv.y, z.x, acc[1][0]); acc[1][1] = fmaf(xv.y, z.y, acc[1][1]);
      acc[1][2] = fmaf(xv.y, z.z, acc[1][2]); acc[1][3] = fmaf(xv.y, z.w, acc[1][3]);
      if (q == 0) {
        bacc[0] += z.x; bacc[1] += z.y; bacc[2] += z.z; bacc[3] += z.w;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int c = c0 + 4 * g + e;
    if (c < K1) {
      atomicAdd(dw_router + (size_t)(i0 + 2 * q) * K1 + c, acc[0][e]);
      atomicAdd(dw_router + (size_t)(i0 + 2 * q + 1) * K1 + c, acc[1][e]);
      if (dbias && blockIdx.x == 0 && q == 0) atomicAdd(dbias + c, bacc[e]);
    }
  }
}

// W*^T: the router's first K+1 columns (fp32 [d][Cp]) as [K+1][d].
__global__ void router_transpose_kernel(int K1, int d, int Cp, const float* __restrict__ wr,
                                        float* __restrict__ wrT) {
  grid_dep_wait();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < K1 * d) {
    const int c = k / d, i = k % d;
    wrT[k] = wr[(size_t)i * Cp + c];
  }
}

// Gram regulariser (Eq. diversity-loss): A = W*^T W* - I over the K+1
// router columns (one block per entry, reduced over d), then L_div = ||A||_F
// and dW* += lambda 2 W* A / L_div (nothing where L_div = 0), W*^T as
// [K+1][d] fp32.
__global__ void __launch_bounds__(128)
gram_kernel(int K1, int d, const float* __restrict__ wrT, float* __restrict__ A) {
  __shared__ float red[4];
  grid_dep_wait();
  const int a = blockIdx.x / K1, b = blockIdx.x % K1;
  float g = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x)
    g = fmaf(wrT[(size_t)a * d + i], wrT[(size_t)b * d + i], g);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = g;
  __syncthreads();
  if (threadIdx.x == 0) A[blockIdx.x] = red[0] + red[1] + red[2] + red[3] - (a == b ? 1.f : 0.f);
}

__global__ void __launch_bounds__(256)
diversity_grad_kernel(int K1, int d, const float* __restrict__ wrT, const float* __restrict__ A,
                      float lambda, float* __restrict__ dw_router, float* __restrict__ l_out) {
  __shared__ float red[8];
  grid_dep_wait();
  float ss = 0.f;
  for (int k = threadIdx.x; k < K1 * K1; k += blockDim.x) ss = fmaf(A[k], A[k], ss);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) tot += red[w];
  const float L = sqrtf(tot);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0 && l_out) *l_out = L;
  if (k >= d * K1 || !(L > 0.f) || lambda == 0.f || !dw_router) return;
  const int i = k / K1, b = k % K1;
  float g = 0.f;
  for (int a = 0; a < K1; ++a) g = fmaf(wrT[(size_t)a * d + i], A[a * K1 + b], g);
  dw_router[k] += 2.f * lambda / L * g;
}

// out[e][c][r] = in[e][r][c] for bf16 [E][R][C] (32 x 32 tiles through shared
// memory).
__global__ void transpose_bf16_kernel(const __nv_bfloat16* __restrict__ in,
                                      __nv_bfloat16* __restrict__ out, int R, int C) {
  __shared__ __nv_bfloat16 tile[32][33];
  const size_t base = (size_t)blockIdx.z * R * C;
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int r = r0 + k, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[k][threadIdx.x] = in[base + (size_t)r * C + c];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int c = c0 + k, r = r0 + threadIdx.x;
    if (r < R && c < C) out[base + (size_t)c * R + r] = tile[threadIdx.x][k];
  }
}

}  // namespace bwd
}  // namespace tc

// ---- host side ----

int backward_setup(unif_moe_layer* L) {
  using namespace tc::bwd;
  const uint64_t E = (uint64_t)L->K + 1;
  Workspace& w = L->ws;
  if (!encode_bf16_map(&L->tm_wdownT, w.w_downT, L->d, E * L->H, tc::kBK, L->up_bn / 2, 128) ||
      !encode_bf16_map(&L->tm_wup_half, L->w_up, L->d, E * L->H, tc::kBK, L->up_bn / 2, 128) ||
      !encode_bf16_map(&L->tm_wupT, w.w_upT, L->H, E * L->d, tc::kBK, L->down_bn, 128) ||
      (L->down_ws && !encode_bf16_map(&L->tm_wupT_ws, w.w_upT, L->H, E * L->d, tc::kBK,
                                      (uint32_t)L->ws_down_bn, 128)) ||
      !encode_bf16_map(&L->tm_da, w.da, L->M, (uint64_t)L->max_rows, tc::kBK, tc::kBM, 128) ||
      !encode_bf16_map(&L->tm_da_st, w.da, L->M, (uint64_t)L->max_rows, 32, 32, 64) ||
      !encode_bf16_map(&L->tm_hw_st, w.hw, L->M, (uint64_t)L->max_rows, 32, 32, 64) ||
      !encode_bf16_map(&L->tm_da_q, w.da, L->M, (uint64_t)L->max_rows, tc::kBK, kRows, 128) ||
      !encode_bf16_map(&L->tm_hw_q, w.hw, L->M, (uint64_t)L->max_rows, tc::kBK, kRows, 128)) {
    set_error("cuTensorMapEncodeTiled failed for the backward maps");
    return UNIF_MOE_ERR_CUDA;
  }
  L->bwd_hidden_stages = kHGather;
  while (L->bwd_hidden_stages > kHMinStages &&
         hidden_smem_bytes(L->up_bn, L->bwd_hidden_stages, L->G) > 232448)
    --L->bwd_hidden_stages;
  L->bwd_hidden_smem = hidden_smem_bytes(L->up_bn, L->bwd_hidden_stages, L->G);
  L->bwd_wgrad_stages = kWStages;
  while (L->bwd_wgrad_stages > kWMinStages &&
         wgrad_smem_bytes(L->up_bn, L->bwd_wgrad_stages, L->G) > 232448)
    --L->bwd_wgrad_stages;
  L->bwd_wgrad_smem = wgrad_smem_bytes(L->up_bn, L->bwd_wgrad_stages, L->G);
  if (L->bwd_hidden_smem > 232448 || L->bwd_wgrad_smem > 232448) {
    set_error("backward: shared memory for block width %d and %d groups exceeds 227 KB", L->M,
              L->G);
    return UNIF_MOE_ERR_SHAPE;
  }
  if (allow_smem(bwd_hidden_kernel, L->bwd_hidden_smem) != cudaSuccess ||
      allow_smem(bwd_wgrad_kernel, L->bwd_wgrad_smem) != cudaSuccess) {
    set_error("cudaFuncSetAttribute failed for the backward kernels");
    return UNIF_MOE_ERR_CUDA;
  }
  return UNIF_MOE_OK;
}

cudaError_t launch_transpose_weights(unif_moe_layer* L, cudaStream_t s) {
  using namespace tc::bwd;
  const int E = L->K + 1;
  dim3 blk(32, 8);
  // w_up [E][H][d] -> w_upT [E][d][H]; w_down [E][d][H] -> w_downT [E][H][d]
  transpose_bf16_kernel<<<dim3((L->d + 31) / 32, (L->H + 31) / 32, E), blk, 0, s>>>(
      static_cast<const __nv_bfloat16*>(L->w_up), static_cast<__nv_bfloat16*>(L->ws.w_upT), L->H,
      L->d);
  transpose_bf16_kernel<<<dim3((L->H + 31) / 32, (L->d + 31) / 32, E), blk, 0, s>>>(
      static_cast<const __nv_bfloat16*>(L->w_down), static_cast<__nv_bfloat16*>(L->ws.w_downT),
      L->d, L->H);
  return cudaGetLastError();
}

int backward_run(unif_moe_layer* L, const void* x, const void* dy, int T, const uint8_t* mask,
                 float* dx, float* dw_up, float* dw_down, float* dw_router, float* dbias,
                 float lambda_div, float* l_div, cudaStream_t s) {
  using namespace tc::bwd;
  Workspace& w = L->ws;
  const int K1 = L->K + 1;
#define CKB(call)                                                               \
  do {                                                                          \
    cudaError_t e_ = (call);                                                    \
    if (e_ != cudaSuccess) {                                                    \
      set_error("%s failed: %s", #call, cudaGetErrorString(e_));                \
      return UNIF_MOE_ERR_CUDA;                                                 \
    }                                                                           \
  } while (0)
  // tile list of the forward's groups (sizes in grp_cnt, rows in the regions);
  // dL/dalpha and dL/ds start at zero
  CKB(launch_tile_list_from(L, w.grp_cnt, w.dwt, (size_t)T * K1, s));
  // hidden gradients
  {
    HiddenParams p;
    p.counts = w.grp_cnt; p.G = L->G; p.region = L->region_rows;
    p.row_tok = w.row_tok; p.row_w = w.row_w;
    p.x = static_cast<const __nv_bfloat16*>(x);
    p.dy = static_cast<const __nv_bfloat16*>(dy);
    p.dwt = w.dwt;
    p.dw_up = dw_up; p.dw_down = dw_down;
    p.w_parts = L->d / 128 * L->up_nsub * 2; p.w_ctas = L->n_sm;
    p.dw_router = dw_router; p.n_wr = L->d * K1;
    p.dbias = dbias; p.n_bias = dbias ? K1 : 0;
    p.n_sub = L->up_nsub; p.bn = L->up_bn; p.num_kb = L->d / tc::kBK;
    p.B = L->B; p.M = L->M; p.H = L->H; p.d = L->d; p.K1 = K1;
    p.stages = L->bwd_hidden_stages;
    p.status = w.status;
    p.wait_limit = gemm_wait_limit();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L->n_sm / 2 * 2);  // a pair per two SMs
    cfg.blockDim = dim3(kHThreads);
    cfg.dynamicSmemBytes = L->bwd_hidden_smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CKB(cudaLaunchKernelEx(&cfg, bwd_hidden_kernel, L->tm_wup_half, L->tm_wdownT, L->tm_da_st,
                           L->tm_hw_st, p));
  }
  // router: W*^T, then dL/dz and its share of dL/dx, which dL/dx starts from
  CKB(launch_dependent(router_transpose_kernel, dim3((K1 * L->d + 255) / 256), dim3(256), 0, s, K1,
                       L->d, L->router_cols_pad, static_cast<const float*>(L->wr), w.wrT));
  {
    const int adaptive = isnan(L->th.alpha_fixed) ? 1 : 0;
    auto dz = K1 <= 16 ? router_dz_kernel<16>
                       : (K1 <= 32 ? router_dz_kernel<32> : router_dz_kernel<65>);
    CKB(launch_dependent(dz, dim3((T + 255) / 256), dim3(256), 0, s, T, L->K, L->tau, adaptive,
                         mask, static_cast<const float*>(w.alpha), static_cast<const float*>(w.s),
                         static_cast<const float*>(w.dwt), w.dz));
    const int items = (T + 1) / 2 * (L->d / 8);
    CKB(launch_dependent(router_dx_kernel, dim3(std::min((items + 255) / 256, 8 * L->n_sm)),
                         dim3(256), 0, s, T, K1, L->d, static_cast<const float*>(w.dz),
                         static_cast<const float*>(w.wrT), dx));
  }
  // dL/dx from the experts: DA K_e (the down kernel on the transposed keys)
  // (weight-stationary where the forward's down projection is: ViT-S, 12,608
  // tokens, 82 -> 71 us)
  if (L->down_ws && T >= kWsTokens)
    CKB(launch_down_ws_on(L, L->tm_da, L->tm_wupT_ws, dx, s));
  else
    CKB(launch_down_streaming(L, L->tm_da, L->tm_wupT, nullptr, dx, s));
  // dL/dK_e and dL/dV_e (chunks of each group's rows add their parts)
  {
    WgradParams p;
    p.counts = w.grp_cnt; p.row_tok = w.row_tok;
    p.x = static_cast<const __nv_bfloat16*>(x);
    p.dy = static_cast<const __nv_bfloat16*>(dy);
    p.dw_up = dw_up; p.dw_down = dw_down;
    p.G = L->G; p.region = L->region_rows; p.B = L->B; p.M = L->M; p.H = L->H; p.d = L->d;
    p.N = L->up_bn; p.n_nc = L->up_nsub; p.n_c = L->d / 128;
    p.stages = L->bwd_wgrad_stages;
    p.status = w.status;
    p.wait_limit = gemm_wait_limit();
    CKB(launch_dependent(bwd_wgrad_kernel, dim3(L->n_sm), dim3(kWThreads), L->bwd_wgrad_smem, s,
                         L->tm_da_q, L->tm_hw_q, p));
  }
  // dL/dW* and dL/dbias
  CKB(launch_dependent(router_dw_kernel,
                       dim3(L->d / 128, (T + kRwSlice - 1) / kRwSlice, (K1 + 15) / 16), dim3(256),
                       0, s, T, K1, L->d, mask, static_cast<const __nv_bfloat16*>(x),
                       static_cast<const float*>(w.dz), dw_router, dbias));
  if (lambda_div != 0.f || l_div) {
    CKB(launch_dependent(gram_kernel, dim3(K1 * K1), dim3(128), 0, s, K1, L->d,
                         static_cast<const float*>(w.wrT), w.gram));
    CKB(launch_dependent(diversity_grad_kernel, dim3((L->d * K1 + 255) / 256), dim3(256), 0, s, K1,
                         L->d, static_cast<const float*>(w.wrT),
                         static_cast<const float*>(w.gram), lambda_div, dw_router, l_div));
  }
#undef CKB
  return UNIF_MOE_OK;
}

}  // namespace unif
