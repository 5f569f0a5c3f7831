// Grouped expert GEMMs on CUDA cores (FP32 FMA), used for fp32 layers: the
// tcgen05 tf32 kind rounds operands to 10 mantissa bits, which an fp32 layer
// cannot afford, so fp32 layers keep full-precision FMA.
//
// Both kernels walk the same tile list as the tensor-core path:
//   up   : h[row] = GeLU(x[tok(row)] K_e[:, H_b])           (Eq. 16, inner part)
//   down : y[tok(row)] += w(row) * h[row] V_e[H_b, :]       (Eqs. 16, 28-30)
// where (e, b) is the tile's group and w(row) is alpha or p_i.
#include "internal.cuh"
#include "items.cuh"

namespace unif {
namespace {

// A 32-row quarter of a 128-row tile x 64 output columns per work item, 128
// threads of 4 x 4 outputs. Small fp32 layers are bound by latency and by
// how many SMs have work (256 tokens of the d = 64 layer: about 20 group
// tiles), so the items are small, the operand tiles of 32 reduction elements
// come through a two-deep cp.async ring, and each 16-byte shared-memory read
// feeds 4 FMAs per row or column. Measured against 128 x 64 items with
// scalar loads into one buffer (both projections, 256 tokens, d = 64, H =
// 256, K = 4, B = 4): 42 -> 14 us.
constexpr int kTM = 32, kTN = 64, kTK = 32, kThreads = 128;
constexpr int kLd = kTK + 4;  // row stride: 16-byte rows, conflict-free float4 column reads

__device__ __forceinline__ float gelu_erf(float v) {
  return 0.5f * v * (1.0f + erff(v * 0.70710678118654752f));
}

struct SimtArgs {
  const int32_t* n_tiles;
  const int32_t* tile_group;
  const int32_t* tile_row0;
  const int32_t* tile_rows;
  const int32_t* row_tok;
  const float* row_w;
  int d, H, B, M;
  int vec;  // every weight row of a block starts on a 16-byte boundary (M % 4 == 0)
  float* y32;
};

__device__ __forceinline__ void cp_async16_zfill(float* dst, const float* src, bool real) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = real ? 16 : 0;  // 0: the 16 bytes are filled with zeros, src is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n)
               : "memory");
}

// MODE 0: up-projection + GeLU into h. MODE 1: down-projection, weighted,
// accumulated into y32 with atomics.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
simt_gemm_kernel(const float* __restrict__ A, const float* __restrict__ W, float* __restrict__ h,
                 SimtArgs a) {
  __shared__ __align__(16) float As[2][kTM][kLd];
  __shared__ __align__(16) float Ws[2][kTN][kLd];
  __shared__ int tok_s[kTM];
  __shared__ float w_s[kTM];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int N = (MODE == 0) ? a.M : a.d;     // output columns of the group
  const int Kdim = (MODE == 0) ? a.d : a.M;  // reduction length
  const bool vec = MODE == 0 || a.vec;       // (d % 8 == 0: rows of x and of w_up are aligned)
  const int n_chunks = (N + kTN - 1) / kTN;
  grid_dep_launch();
  grid_dep_wait();  // the tile list, the rows and (down) h are complete
  const int n_tiles = a.n_tiles[0];
  ItemWalk item(blockIdx.x, gridDim.x, 4 * n_chunks);
  for (; item.tile < n_tiles; item.next()) {
    const int tile = item.tile, q = item.part / n_chunks, n0 = item.part % n_chunks * kTN;
    const int rows = min(kTM, a.tile_rows[tile] - kTM * q);
    if (rows <= 0) continue;  // padding only
    const int g = a.tile_group[tile], row0 = a.tile_row0[tile] + kTM * q;
    const int e = g / a.B, blk = g % a.B;
    // w_up [(K+1)H][d]: row e H + blk M + n; w_down [(K+1)d][H]: row e d + n, column blk M + k
    const float* Wg = MODE == 0 ? W + ((size_t)e * a.H + (size_t)blk * a.M) * a.d
                                : W + (size_t)e * a.d * a.H + (size_t)blk * a.M;
    const int ldw = MODE == 0 ? a.d : a.H;
    __syncthreads();  // the previous item's epilogue has read tok_s and w_s
    if (tid < kTM) {
      tok_s[tid] = tid < rows ? a.row_tok[row0 + tid] : -1;
      w_s[tid] = tid < rows ? a.row_w[row0 + tid] : 0.f;
    }
    __syncthreads();
    // row r of the item is x[tok] (up) or h[row0 + r] (down)
    const float* arow[2];
    bool areal[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = (tid >> 3) + 16 * i, t = tok_s[r];
      areal[i] = t >= 0;
      arow[i] = MODE == 0 ? A + (size_t)max(t, 0) * a.d : A + (size_t)(row0 + r) * a.M;
    }
    const int kc = (tid & 7) * 4;
    auto load = [&](int k0, int buf) {
      if (vec) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const bool real = areal[i] && k0 + kc < Kdim;
          cp_async16_zfill(&As[buf][(tid >> 3) + 16 * i][kc], real ? arow[i] + k0 + kc : A, real);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = (tid >> 3) + 16 * i;
          const bool real = n0 + n < N && k0 + kc < Kdim;
          cp_async16_zfill(&Ws[buf][n][kc], real ? Wg + (size_t)(n0 + n) * ldw + k0 + kc : W,
                           real);
        }
      } else {  // down projection of blocks whose width is no multiple of 4
#pragma unroll
        for (int i = 0; i < 2; ++i)
          for (int j = 0; j < 4; ++j)
            As[buf][(tid >> 3) + 16 * i][kc + j] =
                areal[i] && k0 + kc + j < Kdim ? arow[i][k0 + kc + j] : 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          for (int j = 0; j < 4; ++j) {
            const int n = (tid >> 3) + 16 * i;
            Ws[buf][n][kc + j] = n0 + n < N && k0 + kc + j < Kdim
                                     ? Wg[(size_t)(n0 + n) * ldw + k0 + kc + j] : 0.f;
          }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    load(0, 0);
    for (int k0 = 0, buf = 0; k0 < Kdim; k0 += kTK, buf ^= 1) {
      if (k0 + kTK < Kdim) {
        load(k0 + kTK, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < kTK; kk += 4) {
        float av[4][4], wv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 u = *reinterpret_cast<const float4*>(&As[buf][ty * 4 + i][kk]);
          const float4 v = *reinterpret_cast<const float4*>(&Ws[buf][tx + 16 * i][kk]);
          av[i][0] = u.x; av[i][1] = u.y; av[i][2] = u.z; av[i][3] = u.w;
          wv[i][0] = v.x; wv[i][1] = v.y; wv[i][2] = v.z; wv[i][3] = v.w;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i][m], wv[j][m], acc[i][j]);
      }
      __syncthreads();  // this buffer is loaded again two steps on
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty * 4 + i;
      if (tok_s[r] < 0) continue;  // a padding row's h and output are never read
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = n0 + tx + 16 * j;
        if (n >= N) continue;
        if (MODE == 0)
          h[(size_t)(row0 + r) * a.M + n] = gelu_erf(acc[i][j]);
        else
          atomicAdd(a.y32 + (size_t)tok_s[r] * a.d + n, w_s[r] * acc[i][j]);
      }
    }
  }
}

}  // namespace

cudaError_t launch_gemms_simt(unif_moe_layer* L, const void* x, int T, cudaEvent_t mid,
                              cudaStream_t s) {
  (void)T;
  SimtArgs a;
  a.n_tiles = L->ws.n_tiles; a.tile_group = L->ws.tile_group; a.tile_row0 = L->ws.tile_row0;
  a.tile_rows = L->ws.tile_rows;
  a.row_tok = L->ws.row_tok; a.row_w = L->ws.row_w;
  a.d = L->d; a.H = L->H; a.B = L->B; a.M = L->M; a.y32 = L->ws.y32;
  a.vec = L->M % 4 == 0;
  const int grid = L->n_sm * 4;
  float* h = static_cast<float*>(L->ws.hbuf);
  cudaError_t e = launch_dependent(simt_gemm_kernel<0>, dim3(grid), dim3(kThreads), 0, s,
                                   static_cast<const float*>(x),
                                   static_cast<const float*>(L->w_up), h, a);
  if (e == cudaSuccess && mid) e = cudaEventRecord(mid, s);
  if (e != cudaSuccess) return e;
  // (output: the accumulator)
  return launch_dependent(simt_gemm_kernel<1>, dim3(grid), dim3(kThreads), 0, s,
                          static_cast<const float*>(h), static_cast<const float*>(L->w_down),
                          static_cast<float*>(nullptr), a);
}

}  // namespace unif
