// Rows of the down projection bundled over four blocks (bf16 layers whose
// projections are grouped by (expert, block), many tokens).
//
// Grouped by (expert, block), the down projection adds one fp32 output row
// per pair, C_B rows of d per token (Eq. 35): 2.1 GB of reductions for 12,608
// tokens of the ViT-B layer (K = B = 16), and it ran at exactly the rate of
// its reductions (378 us, 5.6 TB/s; plain adds of the same rows reach
// 6.3). Blocks 4 c .. 4 c + 3 of an expert form bundle c; a token that runs
// expert e there runs a non-empty subset s of the four (its pattern, from
// the shared block set, complemented for a residual expert: Eqs. 23, 28-29).
// The tokens of equal (e, c, s) form a group whose rows go through the
// |s| blocks of s as one reduction of |s| M channels, so that a token adds
// one output row per bundle it touches (24.7 instead of 54.3 on ViT-B) and
// no block is computed that it does not run: 378 -> 268 us, bound by the
// operand bytes out of L2 and the reductions together (without the
// reductions 194). Sharing each tile's h among a cluster of CTAs by TMA
// multicast was slower (497 -> 525 us per forward: 138 of 152 SMs, in
// lockstep), and so were contiguous runs of tiles per CTA (570: neighbouring
// tiles at the same time keep an expert's values in L2). The price is smaller
// groups (15 patterns per bundle), whose last 128-row tiles are partly
// padding: bundles_apply.
//
// h keeps its rows of M channels: the tiles of all bundle groups are numbered
// in units of 128 rows x M, |s| units per tile (one per block of s, in
// order), and the up projection, whose own groups stay (expert, block),
// writes each row to the place that dst names.
#include <math.h>

#include <algorithm>

#include "decide.cuh"
#include "internal.cuh"

namespace unif {
namespace {

constexpr int kPatterns = (1 << kBundle) - 1;  // non-empty subsets of a bundle's blocks
constexpr int kRowsThreads = 256;
constexpr int kRowsTokens = 128;  // tokens per CTA of bundle_rows_kernel, two threads each
constexpr int kTilesThreads = 1024;

struct RowsArgs {
  const uint64_t* shr;
  const uint64_t* em;
  const float* alpha;
  const float* s;  // [T][K]
  int T, K, B, G, region;
  int32_t* fill;     // [G] rows per group, 0 before this pass
  int2* rows;        // [G][region] (token, weight)
  int* status;
};

// Each group's rows (token, weight), in its region, in the order in which the
// CTAs reserve them (one atomic per CTA and group; within a CTA through
// shared-memory cursors). Two threads share a token's experts, four bundles at
// a time (independent cursor updates). A row is one 8-byte store: the groups
// are too many for runs, and every row's sector leaves the SM by itself (two
// 4-byte stores and one bundle after the other: 11.5 us for 12,608 tokens of
// ViT-B, now 10.2; 32,768 tokens of K = 32 14.5, now 13.4).
__global__ void __launch_bounds__(kRowsThreads) bundle_rows_kernel(RowsArgs a) {
  extern __shared__ int32_t cur[];  // [G] this CTA's rows, then its next row
  for (int g = threadIdx.x; g < a.G; g += kRowsThreads) cur[g] = 0;
  grid_dep_wait();  // the router's decisions
  __syncthreads();
  const int t = blockIdx.x * kRowsTokens + (threadIdx.x & (kRowsTokens - 1));
  const int half = threadIdx.x / kRowsTokens;
  const int Q = a.B / kBundle;
  const uint64_t full = a.B >= 64 ? ~0ull : ((1ull << a.B) - 1ull);
  const uint64_t kfull = a.K >= 64 ? ~0ull : ((1ull << a.K) - 1ull);
  const uint64_t shr = t < a.T ? a.shr[t] & full : 0ull;
  // (padding tokens have neither shared blocks nor experts)
  uint64_t em = t < a.T ? a.em[t] & kfull : 0ull;
  em &= half == 0 ? 0x5555555555555555ull : 0xAAAAAAAAAAAAAAAAull;
  const uint64_t comp = ~shr & full;
  // the groups of expert e's bundles, four at a time (-1: none)
  auto bundles = [&](int e, uint64_t blocks, auto&& f) {
    for (int c0 = 0; c0 < Q; c0 += 4) {
      const uint32_t b16 = (uint32_t)(blocks >> (kBundle * c0)) & 0xffffu;
      int g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int s = (int)(b16 >> (kBundle * u)) & kPatterns;
        g[u] = s ? (e * Q + c0 + u) * kPatterns + s - 1 : -1;
      }
      f(g);
    }
  };
  auto count = [&](const int (&g)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (g[u] >= 0) atomicAdd(&cur[g[u]], 1);
  };
  if (half == 0) bundles(0, shr, count);
  for (uint64_t r = em; r != 0ull; r &= r - 1ull) bundles(__ffsll((long long)r), comp, count);
  __syncthreads();
  // reservations, four groups' atomics in flight per thread
  for (int g0 = threadIdx.x; g0 < a.G; g0 += 4 * kRowsThreads) {
    int n[4], base[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) n[u] = g0 + u * kRowsThreads < a.G ? cur[g0 + u * kRowsThreads] : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) base[u] = n[u] > 0 ? atomicAdd(a.fill + g0 + u * kRowsThreads, n[u]) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (n[u] > 0) {
        if (base[u] + n[u] > a.region) {  // stale counters: stay inside the region
          atomicOr(a.status, kStatusBadIndex);
          base[u] = a.region;
        }
        cur[g0 + u * kRowsThreads] = base[u];
      }
  }
  __syncthreads();
  float w = 0.f;
  auto place = [&](const int (&g)[4]) {
    int p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) p[u] = g[u] >= 0 ? atomicAdd(&cur[g[u]], 1) : a.region;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p[u] < a.region)
        a.rows[(size_t)g[u] * a.region + p[u]] = make_int2(t, __float_as_int(w));
  };
  // (an expert's weight is on its way while the one before is placed)
  auto weight = [&](uint64_t r) {
    return r != 0ull ? a.s[(size_t)t * a.K + __ffsll((long long)r) - 1] : 0.f;
  };
  float w_nxt = weight(em);
  if (half == 0 && shr != 0ull) {
    w = a.alpha[t];
    bundles(0, shr, place);
  }
  for (uint64_t r = em; r != 0ull; r &= r - 1ull) {
    w = w_nxt;
    w_nxt = weight(r & (r - 1ull));
    bundles(__ffsll((long long)r), comp, place);
  }
}

struct TilesArgs {
  const int32_t* fill;
  const int2* rows;
  int G, region, Q, K1;
  int32_t* n_tiles;
  int32_t* tile_group;
  int32_t* tile_row0;
  int32_t* tile_rows;
  int32_t* tile_unit;
  int32_t* dst;
};

// The 128-row tiles of the groups (group, first list row, real rows, first
// unit of h) and dst[(t (K + 1) + e) Q + c]: the h row of token t's first
// block in bundle c of expert e (its i-th block's is 128 i rows on). Every
// CTA scans the group sizes for itself; a warp per tile.
__global__ void __launch_bounds__(kTilesThreads) bundle_tiles_kernel(TilesArgs a) {
  extern __shared__ int32_t sm[];  // [G + 1] first tiles, [G] first units, [G] sizes
  __shared__ int2 wsum[kTilesThreads / 32];
  int32_t* first_t = sm;
  int32_t* first_u = first_t + a.G + 1;
  int32_t* cnt = first_u + a.G;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  grid_dep_wait();  // the groups' rows
  const int per = (a.G + kTilesThreads - 1) / kTilesThreads;
  const int ga = min(a.G, tid * per), gb = min(a.G, ga + per);
  auto blocks = [](int g) { return __popc(g % kPatterns + 1); };
  int2 mine = make_int2(0, 0);  // tiles, units
  for (int g = ga; g < gb; ++g) {
    const int c = min(__ldcg(a.fill + g), a.region), nt = (c + kTileRows - 1) / kTileRows;
    cnt[g] = c;
    mine.x += nt;
    mine.y += nt * blocks(g);
  }
  int2 inc = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, inc.x, o), y = __shfl_up_sync(0xffffffffu, inc.y, o);
    if (lane >= o) {
      inc.x += x;
      inc.y += y;
    }
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  int2 base = make_int2(inc.x - mine.x, inc.y - mine.y);
  for (int w = 0; w < warp; ++w) {
    base.x += wsum[w].x;
    base.y += wsum[w].y;
  }
  for (int g = ga; g < gb; ++g) {
    first_t[g] = base.x;
    first_u[g] = base.y;
    const int nt = (cnt[g] + kTileRows - 1) / kTileRows;
    base.x += nt;
    base.y += nt * blocks(g);
  }
  if (tid == kTilesThreads - 1) first_t[a.G] = base.x;
  __syncthreads();
  const int nt = first_t[a.G];
  if (blockIdx.x == 0 && tid == 0) a.n_tiles[0] = nt;
  for (int k = blockIdx.x * (kTilesThreads / 32) + warp; k < nt;
       k += gridDim.x * (kTilesThreads / 32)) {
    int lo = 0, hi = a.G - 1;  // the last group whose first tile is <= k
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first_t[mid] <= k) lo = mid; else hi = mid - 1;
    }
    const int i = k - first_t[lo];
    const int row0 = lo * a.region + kTileRows * i, rows = min(kTileRows, cnt[lo] - kTileRows * i);
    const int unit = first_u[lo] + i * blocks(lo);
    if (lane == 0) {
      a.tile_group[k] = lo;
      a.tile_row0[k] = row0;
      a.tile_rows[k] = rows;
      a.tile_unit[k] = unit;
    }
    const int ec = lo / kPatterns, e = ec / a.Q, c = ec % a.Q;
    for (int r = lane; r < rows; r += 32)
      a.dst[((size_t)a.rows[row0 + r].x * a.K1 + e) * a.Q + c] = unit * kTileRows + r;
  }
}

}  // namespace

// Bundles can be used by a layer: its up projection is the pair kernel's,
// whole bundles, tables that fit in shared memory, list indexes within int32.
bool bundles_fit(const unif_moe_layer* L) {
  const int64_t G = (int64_t)(L->K + 1) * (L->B / kBundle) * kPatterns;
  return L->fused_group && !L->ffn_fused && !L->gemm_streaming && up_ws_bytes(L) == 0 &&
         L->B % kBundle == 0 && G <= 4096 && G * L->region_rows < ((int64_t)1 << 31) &&
         (int64_t)L->pass_tokens * (L->K + 1) * (L->B / kBundle) < ((int64_t)1 << 31) &&
         bundle_h_rows(L) < ((int64_t)1 << 31);
}

int bundle_groups(const unif_moe_layer* L) {
  return (L->K + 1) * (L->B / kBundle) * kPatterns;
}

// h rows: at most the pairs of a pass plus 127 padding rows per block of every
// group, and room for a stale dst.
int64_t bundle_h_rows(const unif_moe_layer* L) {
  const int64_t padded = (int64_t)(L->K + 1) * (L->B / kBundle) * (kBundle << (kBundle - 1));
  const int64_t rows = (int64_t)L->pass_tokens * L->cb_max + padded * (kTileRows - 1);
  return (rows + kTileRows - 1) / kTileRows * kTileRows + (int64_t)kBundle * kTileRows;
}

int64_t bundle_max_tiles(const unif_moe_layer* L) {
  const int64_t kmax = L->cb_max / L->B;
  const int64_t rows = (int64_t)L->pass_tokens * (1 + kmax) * (L->B / kBundle);
  return rows / kTileRows + bundle_groups(L) + 1;
}

// A pass of T tokens bundles its rows where the groups hold at least M^2 / 500
// tokens on average: T (1 + k) / (K + 1) tokens per expert over 15 patterns, k
// the fixed count or else about K / 3, or 2/3 beta K where a fixed mass (beta,
// or 1 - alpha) makes it less. Narrow blocks gain most (an output
// row per M channels of work), and small groups lose to padding. Measured, us
// per forward without and with bundles: d = 768, K = 16, M = 192: 2,500
// tokens (62 per group) 167 and 172, 4,000 228 and 203, 12,608 583 and 497;
// with two experts per token 5,000 (59) 153 and 168, 12,608 288 and 250; with
// beta = 0.05 3,000 (24) 89 and 139, 6,000 135 and 162, 12,608 219 and 218; with
// alpha = 0.9 3,000 102 and 118, 6,000 146 and 145, 12,608 220 and 199; K =
// 10, M = 256: 4,000 (105) 163 and 149; K = 8, M = 384: 7,000 (190) 172 and
// 177, 14,000 319 and 305; d = 1024, skewed, K = 32, M = 256: 6,000 (141) 412
// and 415, 9,000 546 and 502; K = 12, M = 512: 20,000 (512) 414 and 420.
// T counts padding too, which the host does not know: half-padded batches near
// the line lose a little (3,000 slots of the first layer 132 and 154).
bool bundles_apply(const unif_moe_layer* L, int T) {
  if (!L->bundles) return false;
  const unif_moe_thresholds& th = L->th;
  double k = L->K / 3.0;
  if (th.topk_fixed > 0) {
    k = th.topk_fixed;
  } else if (!isnan(th.beta_fixed) || !isnan(th.alpha_fixed)) {
    const double beta = isnan(th.beta_fixed) ? 1.0 - th.alpha_fixed : th.beta_fixed;
    k = std::min(k, std::max(1.0, 2.0 / 3.0 * beta * L->K));
  }
  return (double)T * (1.0 + k) * 500.0 >= (double)L->M * L->M * kPatterns * (L->K + 1);
}

cudaError_t bundles_setup(const unif_moe_layer* L) {
  return allow_smem(bundle_tiles_kernel, (3 * bundle_groups(L) + 1) * sizeof(int32_t));
}

cudaError_t launch_bundles(unif_moe_layer* L, int T, cudaStream_t s) {
  Workspace& w = L->ws;
  const int G = bundle_groups(L);
  const size_t r0 = (size_t)L->rec0;  // the records of this pass's first token
  RowsArgs r;
  r.shr = w.shr_mask + r0; r.em = w.exp_mask + r0; r.alpha = w.alpha + r0;
  r.s = w.s + r0 * L->K;
  r.T = T; r.K = L->K; r.B = L->B; r.G = G; r.region = L->region_rows;
  r.fill = w.bd_fill; r.rows = w.bd_rows; r.status = w.status;
  cudaError_t e = launch_dependent(bundle_rows_kernel, dim3((T + kRowsTokens - 1) / kRowsTokens),
                                   dim3(kRowsThreads), sizeof(int32_t) * G, s, r);
  if (e != cudaSuccess) return e;
  TilesArgs t;
  t.fill = w.bd_fill; t.rows = w.bd_rows;
  t.G = G; t.region = L->region_rows; t.Q = L->B / kBundle; t.K1 = L->K + 1;
  t.n_tiles = w.bd_n_tiles; t.tile_group = w.bd_tile_group; t.tile_row0 = w.bd_tile_row0;
  t.tile_rows = w.bd_tile_rows; t.tile_unit = w.bd_tile_unit; t.dst = w.bd_dst;
  return launch_dependent(bundle_tiles_kernel, dim3(L->n_sm), dim3(kTilesThreads),
                          sizeof(int32_t) * (3 * G + 1), s, t);
}

}  // namespace unif
