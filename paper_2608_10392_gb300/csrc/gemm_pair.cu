// Up projection on CTA pairs (tcgen05 cta_group::2, M = 256) for bf16 layers
// whose (expert, block) weight slice does not fit in shared memory (d = 768,
// 1024), and for small passes of the others: h[row] = GeLU(x[tok(row)] K_e[:, H_b]) over the router's groups
// (Eq. 16, inner part).
//
// What bounds it: operand bytes out of L2. The single-CTA streaming kernel
// loads 16 KB of gathered x rows and bn x 128 bytes of keys per 64-deep step
// of a 128-row tile; a pair shares the keys of a step between two 128-row
// halves of a 256-row tile, each CTA loading half of them, so a step costs
// each SM 16 KB + bn x 64 bytes (bn = 192: 28 KB instead of 40).
// Measured against the streaming kernel (us per forward): 128 tokens of the
// BERT-base layer 57 -> 45, its sublayer on 4,096 slots 98 -> 87, ViT-B 671 ->
// 586 (this kernel 253 -> 163), 65,536 tokens of d = 1024 3,724 -> 3,348. The
// stores of h account for 28 of the 163 us, the spread of the gathered rows
// for 5; the tensor pipe's share is 115.
//
// Roles (each CTA of the pair, 18 warps):
//   warps 0-7   gather this CTA's 128 x rows of a step (16-byte cp.async into
//               the 128-byte swizzled layout); warp w owns ring stage w and
//               waits for its own copies before it signals them. (A warp with
//               several steps in flight gains nothing: the proxy fence that
//               must follow each step's copies waits for the later ones too,
//               measured 1,200-1,800 cycles per step with four such warps.)
//   warp 8      this CTA's half of the step's keys by TMA
//   warp 9      TMEM allocation (both CTAs); MMA issue (even CTA); the tile
//               list of a streaming down projection (odd CTAs)
//   warps 10-17 epilogue: GeLU, bf16, h rows to device memory (warp w: TMEM
//               lane quarter w % 4, one half of the columns)
// The ring's full barriers are the even CTA's: the stage's owner warp of each
// CTA and the bytes of both key halves. Its commits free the stages and publish the
// accumulators (two, in TMEM) on both CTAs. Every wait is bounded; a wait
// that runs out records kStatusTimeout and the CTA unwinds.
#include <stdio.h>

#include "decide.cuh"
#include "internal.cuh"
#include "tc_common.cuh"

namespace unif {
namespace tc {
namespace pair {

constexpr int kGatherWarps = 8;  // at most one per ring stage
constexpr int kLoaderWarp = 8;
constexpr int kMmaWarp = 9;
constexpr int kFirstEpi = 10;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (kFirstEpi + kEpiWarps);  // 576
constexpr int kPairRows = 256;
constexpr int kMinStages = 5;
constexpr int kMaxStages = kGatherWarps;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAccStride = 256;
constexpr uint32_t kHStageRow = 80;    // bytes per staged h row (64 + 16 pad)
constexpr uint32_t kStaging = kEpiWarps * 32u * kHStageRow;
constexpr uint32_t kBarBytes = 256;
constexpr uint32_t kMaxSmem = 232448;

struct Params {
  const int32_t* fill;     // [G] rows per group (final once the router completed)
  int G, region;           // groups of `region` rows
  const int32_t* row_tok;  // [G][region] pass-relative token of each row
  const __nv_bfloat16* x;  // [T][d]
  __nv_bfloat16* h;        // [128-row tiles of all groups][M]
  int n_sub, bn, num_kb;   // N sub-tiles of bn columns, 64-deep steps
  int B, M, H, d, stages;
  // the streaming down projection's tile list, written here (null: none)
  int32_t* n_tiles;
  int32_t* tile_group;
  int32_t* tile_row0;
  int32_t* tile_rows;
  // SCATTER: the place in h of every row (bundles.cu)
  const uint64_t* shr;     // [T] shared block sets
  const int32_t* dst;      // [T][K+1][B / kBundle]
  int* status;
  long long wait_limit;
};

__host__ __device__ constexpr uint32_t stage_bytes(int bn) { return kStageA + (uint32_t)bn * 64u; }
__host__ __device__ constexpr uint32_t smem_bytes(int bn, int stages, int G) {
  return 1024u + (uint32_t)stages * stage_bytes(bn) + kStaging + kBarBytes +
         (uint32_t)((3 * G + 2) * 4 + 15) / 16u * 16u;
}

// A bounded wait that ignores the abort flag (copies and MMAs in flight land
// before the pair releases its TMEM).
__device__ __forceinline__ void wait_settle(uint32_t bar, uint32_t parity, long long limit) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > limit) return;
}

// SCATTER: h rows go where dst names (the bundled down projection's units);
// otherwise each group's rows fill its 128-row tiles in list order.
template <bool SCATTER>
__global__ void __launch_bounds__(kThreads, 1)
pair_up_kernel(const __grid_constant__ CUtensorMap tmB, Params p) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned base, the same offset in both CTAs of the pair
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int n_st = p.stages;
  const uint32_t st_bytes = stage_bytes(p.bn);
  const uint32_t s0 = smem_u32(smem);
  // stage s: [128 x rows x 64][bn / 2 key rows x 64]
  auto sa = [&](int s) { return s0 + (uint32_t)s * st_bytes; };
  auto sb = [&](int s) { return s0 + (uint32_t)s * st_bytes + kStageA; };
  uint8_t* staging = smem + (size_t)n_st * st_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kStaging);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kMaxStages + s); };
  auto accf_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + a); };
  auto acce_bar = [&](int a) { return bar0 + 8u * (2 * kMaxStages + 2 + a); };
  const uint32_t mma_done = bar0 + 8u * (2 * kMaxStages + 4);
  const uint32_t fin = bar0 + 8u * (2 * kMaxStages + 5);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 6);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert(8 * (2 * kMaxStages + 7) <= kBarBytes, "barrier region");
  // first 256-row pair tile and first 128-row tile of every group, its size
  int32_t* first_s = reinterpret_cast<int32_t*>(reinterpret_cast<uint8_t*>(bars) + kBarBytes);
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
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(full_bar(s), 3);  // an owner warp of each CTA, the leader's loader
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), 2 * kEpiWarps);
    }
    mbar_init(mma_done, 1);
    mbar_init(fin, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish_pair();
  }
  grid_dep_wait();  // the group sizes and rows
  for (int g = threadIdx.x; g < p.G; g += kThreads) cnt_s[g] = min(__ldcg(p.fill + g), p.region);
  __syncthreads();
  if (warp == 0) {
    tile_scan(p.G, lane, first128_s, cnt_s);
  } else if (warp == 1) {
    tile_scan<kPairRows>(p.G, lane, first_s, cnt_s);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  // both CTAs' barriers are initialised before either CTA signals the other
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // (pair tile, sub-tile) items, dealt out in turn: the pairs work on
  // neighbouring tiles of one expert at a time, whose keys and x rows L2
  // then holds
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int n_items = first_s[p.G] * p.n_sub;
  // the last group whose first pair tile is <= tile
  auto group_of = [&](int tile) {
    int lo = 0, hi = p.G - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first_s[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
  };
  // group, sub-tile and this CTA's first row in the group of an item
  struct Item { int g, ns, pos, rows; };
  auto item_of = [&](int item) {
    Item it;
    const int tile = item / p.n_sub;
    it.ns = item - tile * p.n_sub;
    it.g = group_of(tile);
    it.pos = kPairRows * (tile - first_s[it.g]) + kBM * (int)rank;
    it.rows = max(0, min(kBM, cnt_s[it.g] - it.pos));
    return it;
  };

  if (warp < kGatherWarps) {
    // ---------------- this CTA's x rows of the steps of stage `warp` --------
    const int j8 = lane & 7, rsub = lane >> 3;
    const __nv_bfloat16* xj = p.x + j8 * 8;
    const uint32_t dst = sa(warp);
    bool ok = true;
    uint32_t ph = 0;
    int kb = warp;  // this warp's next step, counted from the item's first
    for (int item = pair; item < n_items && ok && warp < n_st; item += n_pairs) {
      if (kb < p.num_kb) {
        const Item it = item_of(item);
        int tok[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          tok[i] = 32 * i + lane < it.rows
                       ? p.row_tok[(size_t)it.g * p.region + it.pos + 32 * i + lane] : -1;
        for (; kb < p.num_kb; kb += n_st) {
          ok = wait_warp(empty_bar(warp), ph ^ 1u, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          ph ^= 1u;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int row = 4 * i + rsub;
            const int t = __shfl_sync(0xffffffffu, tok[i >> 3], row & 31);
            // (padding rows keep whatever the stage holds: their h is not stored)
            if (t >= 0)
              cp_async16(dst + (uint32_t)row * 128u + ((uint32_t)(j8 ^ (row & 7)) << 4),
                         xj + (size_t)t * p.d + kb * kBK);
          }
          cp_async_commit();
          cp_async_wait<0>();
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) arrive_leader(full_bar(warp));
        }
      }
      kb -= p.num_kb;  // steps count on over the items
    }
  } else if (warp == kLoaderWarp) {
    // ---------------- this CTA's half of every step's keys ------------------
    bool ok = true;
    int s = 0;
    uint32_t ph = 0;
    long long issued = 0;
    for (int item = pair; item < n_items && ok; item += n_pairs) {
      const Item it = item_of(item);
      const int e = it.g / p.B, blk = it.g - e * p.B;
      const int row = e * p.H + blk * p.M + it.ns * p.bn + (int)rank * (p.bn / 2);
      for (int kb = 0; kb < p.num_kb; ++kb) {
        ok = wait_warp(empty_bar(s), ph ^ 1u, abort_flag, p.status, p.wait_limit);
        if (!ok) break;
        if (lane == 0) {
          if (leader) mbar_expect_tx(full_bar(s), (uint32_t)p.bn * 128u);
          tma_load_2d_pair(sb(s), &tmB, mapa_shared(full_bar(s), 0), kb * kBK, row);
        }
        __syncwarp();
        ++issued;
        if (++s == n_st) { s = 0; ph ^= 1u; }
      }
    }
    // loads still in flight land before the pair exits
    if (leader && lane == 0)
      for (long long j = issued > n_st ? issued - n_st : 0; j < issued; ++j)
        wait_settle(full_bar((int)(j % n_st)), (uint32_t)((j / n_st) & 1), p.wait_limit / 16);
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ---------------- MMA issue (the leader CTA) ----------------------------
    if (leader) {
      const uint32_t idesc = idesc_bf16(2 * kBM, p.bn);
      const uint16_t both = 3;
      int s = 0, acc = 0;
      uint32_t ph = 0, acc_ph = 0;
      bool ok = true, any = false;
      for (int item = pair; item < n_items && ok; item += n_pairs) {
        ok = wait_warp_cluster(acce_bar(acc), acc_ph ^ 1u, abort_flag, p.status, p.wait_limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * kAccStride;
        for (int kb = 0; kb < p.num_kb; ++kb) {
          ok = wait_warp_cluster(full_bar(s), ph, abort_flag, p.status, p.wait_limit);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t a = sw128_desc(sa(s)), b = sw128_desc(sb(s));
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16_pair(d_tmem, a + 2 * k, b + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            umma_commit_pair(empty_bar(s), both);
            if (kb == p.num_kb - 1) umma_commit_pair(accf_bar(acc), both);
          }
          __syncwarp();
          any = true;
          if (++s == n_st) { s = 0; ph ^= 1u; }
        }
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
      }
      // every MMA issued has completed before the pair releases TMEM
      if (any) {
        if (elect_one()) umma_commit_pair(mma_done, 1);
        __syncwarp();
        wait_settle(mma_done, 0u, p.wait_limit);
      }
    } else if (p.n_tiles != nullptr) {
      // the peer's MMA warp, which has no MMAs to issue, lists the 128-row
      // tiles for the streaming down projection (a kernel of its own took
      // 3.3 us of every forward)
      const int nt = first128_s[p.G];
      if (pair == 0 && lane == 0) *p.n_tiles = nt;
      for (int k = 32 * pair + lane; k < nt; k += 32 * n_pairs) {
        int g, row0, rows;
        tile_lookup(k, first128_s, cnt_s, p.G, p.region, g, row0, rows);
        p.tile_group[k] = g;
        p.tile_row0[k] = row0;
        p.tile_rows[k] = rows;
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: h = bf16(GeLU(U)) ---------------------------
    const int q = warp & 3, half = (warp - kFirstEpi) >> 2;
    const int cols = p.bn / 2, c_begin = half * cols;
    uint8_t* stg = staging + (size_t)(warp - kFirstEpi) * 32 * kHStageRow;
    int acc = 0;
    uint32_t acc_ph = 0;
    // SCATTER: this lane's row of the next item, its token one item ahead
    // and its shared set and place loaded while the current one is stored
    Item it = item_of(min(pair, max(n_items - 1, 0)));
    auto token_of = [&](const Item& m) {
      const int r = 32 * q + lane;
      return r < m.rows ? p.row_tok[(size_t)m.g * p.region + m.pos + r] : 0;
    };
    int tok = 0;
    if (SCATTER && pair < n_items) tok = token_of(it);
    for (int item = pair; item < n_items; item += n_pairs) {
      const int rows = it.rows - q * 32;  // real rows of this quarter
      __nv_bfloat16* hrow0;
      int drow = 0;  // SCATTER: this lane's h row
      Item nx = it;
      if (item + n_pairs < n_items) nx = item_of(item + n_pairs);
      if (SCATTER) {
        const int e = it.g / p.B, blk = it.g - e * p.B, bit = blk % kBundle;
        const uint64_t sh = p.shr[tok];
        const int d0 = p.dst[((size_t)tok * (p.G / p.B) + e) * (p.B / kBundle) + blk / kBundle];
        // the blocks of the bundle before this one that the row runs
        const uint32_t run = (uint32_t)((e == 0 ? sh : ~sh) >> (blk - bit));
        drow = d0 + kBM * __popc(run & ((1u << bit) - 1u));
        tok = token_of(nx);
        hrow0 = p.h + it.ns * p.bn + c_begin;
      } else {
        hrow0 =
            p.h + ((size_t)first128_s[it.g] * kBM + it.pos + q * 32) * p.M + it.ns * p.bn + c_begin;
      }
      it = nx;
      if (!wait_warp(accf_bar(acc), acc_ph, abort_flag, p.status, p.wait_limit)) break;
      tc_fence_after();
      const uint32_t t_row =
          tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)acc * kAccStride + c_begin;
      if (rows > 0) {
        for (int c = 0; c < cols; c += 32) {
          uint32_t v[32];
          tmem_ld32_async(t_row + c, v);
          tmem_wait_ld();
          uint32_t o[16];
#pragma unroll
          for (int jj = 0; jj < 16; ++jj)
            o[jj] = gelu2_bf16x2(__uint_as_float(v[2 * jj]), __uint_as_float(v[2 * jj + 1]));
#pragma unroll
          for (int jj = 0; jj < 4; ++jj)
            *reinterpret_cast<uint4*>(stg + lane * kHStageRow + 16 * jj) =
                make_uint4(o[4 * jj], o[4 * jj + 1], o[4 * jj + 2], o[4 * jj + 3]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 8 * i + (lane >> 2), seg = lane & 3;
            const int hr = SCATTER ? __shfl_sync(0xffffffffu, drow, r) : r;
            if (r < rows)
              *reinterpret_cast<uint4*>(hrow0 + (size_t)hr * p.M + c + seg * 8) =
                  *reinterpret_cast<const uint4*>(stg + r * kHStageRow + 16 * seg);
          }
          __syncwarp();
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_leader(acce_bar(acc));
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
  }
  // every warp converged before the CTA barrier; then each CTA tells its peer
  // that it is done with the pair's TMEM (the leader after its MMAs
  // completed), and the owner warp waits for the peer's word
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) mbar_arrive_cluster(mapa_shared(fin, rank ^ 1u));
  if (warp == kMmaWarp) {
    wait_settle(fin, 0u, p.wait_limit);
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

}  // namespace pair
}  // namespace tc

// Sets the pair kernel up for the up projection, where the ring holds
// kMinStages stages beside the group tables.
int gemm_pair_setup(unif_moe_layer* L) {
  using namespace tc::pair;
  L->up_pair = false;
  if (!L->fused_group || L->gemm_streaming || L->up_bn % 64 != 0) return UNIF_MOE_OK;
  const uint32_t fixed = smem_bytes(L->up_bn, 0, L->G);
  int stages = fixed < kMaxSmem ? (int)((kMaxSmem - fixed) / stage_bytes(L->up_bn)) : 0;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages < kMinStages) return UNIF_MOE_OK;
  L->pair_stages = stages;
  L->pair_smem = smem_bytes(L->up_bn, stages, L->G);
  if (!encode_bf16_map(&L->tm_wup_half, L->w_up, L->d, (uint64_t)(L->K + 1) * L->H, tc::kBK,
                       (uint32_t)L->up_bn / 2, 128) ||
      allow_smem(pair_up_kernel<false>, L->pair_smem) != cudaSuccess ||
      allow_smem(pair_up_kernel<true>, L->pair_smem) != cudaSuccess) {
    set_error("setting up the pair up-projection kernel failed");
    return UNIF_MOE_ERR_CUDA;
  }
  L->up_pair = true;
  return UNIF_MOE_OK;
}

cudaError_t launch_up_pair(unif_moe_layer* L, const void* x, bool list, bool scatter,
                           cudaStream_t s) {
  tc::pair::Params p;
  p.fill = L->ws.grp_fill;
  p.G = L->G;
  p.region = L->region_rows;
  p.row_tok = L->ws.row_tok;
  p.x = static_cast<const __nv_bfloat16*>(x);
  p.h = static_cast<__nv_bfloat16*>(L->ws.hbuf);
  p.n_sub = L->up_nsub; p.bn = L->up_bn; p.num_kb = L->d / tc::kBK;
  p.B = L->B; p.M = L->M; p.H = L->H; p.d = L->d;
  p.stages = L->pair_stages;
  p.n_tiles = list ? L->ws.n_tiles : nullptr;
  p.tile_group = L->ws.tile_group; p.tile_row0 = L->ws.tile_row0; p.tile_rows = L->ws.tile_rows;
  p.shr = L->ws.shr_mask + L->rec0;
  p.dst = L->ws.bd_dst;
  p.status = L->ws.status;
  p.wait_limit = gemm_wait_limit();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(L->n_sm / 2 * 2);  // a pair per two SMs
  cfg.blockDim = dim3(tc::pair::kThreads);
  cfg.dynamicSmemBytes = L->pair_smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return scatter ? cudaLaunchKernelEx(&cfg, tc::pair::pair_up_kernel<true>, L->tm_wup_half, p)
                 : cudaLaunchKernelEx(&cfg, tc::pair::pair_up_kernel<false>, L->tm_wup_half, p);
}

}  // namespace unif
