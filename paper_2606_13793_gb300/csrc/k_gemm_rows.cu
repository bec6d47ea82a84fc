// Neighbour contraction on the CUDA cores for grids of few rows (FP32): the
// coarse M2L levels of every solve, split over the 27 neighbours.
//
//   part_d[r][n] = sum_{k < K(n)} A[r + d][k] W_d[k][n],  C = sum_d part_d
//
// Each sum runs over k in order and the partials are added in neighbour order,
// one rounding per step: the order of the 4 x 4 x 4 tile's split form, which it
// replaced (those levels carry the bulk of phi, and the 5-point force amplifies
// any change of their rounding).
//
// These levels (8, 64, 512 rows) are bound by latency: a chain of up to
// 8 (p+1)^2 multiply-adds per output, and a kernel each.  So: one launch for
// all of a plan's coarse levels; one warp per (32 rows x 32 columns,
// neighbour), a CTA of its own, so that the long column tiles, first in the
// grid, spread over all SMs; its operands by double-buffered 16-byte cp.async
// in chunks of 32 values of k; a 4 x 8 register tile per lane, cut to the
// live rows of the block.  Levels 2-4 at p = 6, launch by launch: 540 us as
// three 4 x 4 x 4 launches, 56 us as one with 64 rows and four warps a CTA;
// whole 64^3 solve 112 us so, 116 us with one warp a CTA, 107 us with 32 rows
// and four, 105 us with 32 rows and one (12 warps an SM instead of 8, and the
// longest chain of multiply-adds halved).
#include "fmm_internal.h"

namespace fmmgb {
namespace {

constexpr int kRwRows = 32;    // rows per warp
constexpr int kRwTR = kRwRows / 8;  // rows per lane
constexpr int kRwKC = 32;      // reduction values per stage
constexpr int kRwPitch = kRwKC + 4;
constexpr int kRwStage = kRwRows * kRwPitch + kRwKC * kNTile;  // floats
constexpr size_t kRwSmem = sizeof(float) * 2 * kRwStage;

struct RowsGroup {
  NbrGemm g[kRowsGroupMax];
  int first[kRowsGroupMax + 1];  // first item (row block, neighbour) of each level; the reduction: first block
  int n;
};

__device__ __forceinline__ void rw_cp16(float* dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ unsigned long long rw_fma2(unsigned long long a, unsigned long long b,
                                                      unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long rw_splat(float a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}

// One stage: rows rg + 8 i (i < TR), columns 8 cg .. 8 cg + 7, k ascending.
template <int TR>
__device__ __forceinline__ void rw_stage(const float* As, const float* Ws, int kn, int rg, int cg,
                                         unsigned long long (&acc)[kRwTR][4]) {
  for (int k0 = 0; k0 < kn; k0 += 4) {
    float4 a[TR];
#pragma unroll
    for (int i = 0; i < TR; ++i) a[i] = *reinterpret_cast<const float4*>(As + (rg + 8 * i) * kRwPitch + k0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ulonglong2* w = reinterpret_cast<const ulonglong2*>(Ws + (k0 + k) * kNTile + cg * 8);
      const ulonglong2 w0 = w[0], w1 = w[1];
#pragma unroll
      for (int i = 0; i < TR; ++i) {
        const unsigned long long v = rw_splat(k == 0 ? a[i].x : k == 1 ? a[i].y : k == 2 ? a[i].z : a[i].w);
        acc[i][0] = rw_fma2(v, w0.x, acc[i][0]);
        acc[i][1] = rw_fma2(v, w0.y, acc[i][1]);
        acc[i][2] = rw_fma2(v, w1.x, acc[i][2]);
        acc[i][3] = rw_fma2(v, w1.y, acc[i][3]);
      }
    }
  }
}

__global__ void __launch_bounds__(32) nbr_gemm_rows_kernel(const __grid_constant__ RowsGroup G, int per_tile) {
  extern __shared__ __align__(16) float rw_smem[];
  const int lane = threadIdx.x, item = (int)blockIdx.x;
  const int tile = item / per_tile;  // longest reductions first
  int rem = item - tile * per_tile, li = 0;
  while (li + 1 < G.n && rem >= G.first[li + 1]) ++li;
  rem -= G.first[li];
  const NbrGemm& g = G.g[li];
  const int rows = g.grid[0] * g.grid[1] * g.grid[2];
  const int d = rem % 27, r0 = rem / 27 * kRwRows;
  if (d == 13 && g.skip_center) return;  // zero, and left out of the reduction
  const int live = min(kRwRows, rows - r0);
  const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
  const int K = g.tile_k[tile];
  const float* W = static_cast<const float*>(g.W) + g.tile_w[tile] + (long long)d * K * kNTile;
  const float* A = static_cast<const float*>(g.A);
  float* st = rw_smem;

  // this lane's 16-byte pieces: rows (lane / 8) + 4 i, piece lane % 8 of each
  const int q = lane & 7;
  int off[kRwRows / 4];  // source row, -1 outside the grid
#pragma unroll
  for (int i = 0; i < kRwRows / 4; ++i) {
    const int r = r0 + (lane >> 3) + 4 * i;
    const int x = r % g.grid[0] + dx, y = (r / g.grid[0]) % g.grid[1] + dy, z = r / (g.grid[0] * g.grid[1]) + dz;
    off[i] = (r < rows && x >= 0 && y >= 0 && z >= 0 && x < g.grid[0] && y < g.grid[1] && z < g.grid[2])
                 ? (z * g.grid[1] + y) * g.grid[0] + x
                 : -1;
  }
  auto load = [&](int kc, float* s) {
    if (kc < K) {
      const int kn = min(kRwKC, K - kc);
      if (q * 4 < kn) {
#pragma unroll
        for (int i = 0; i < kRwRows / 4; ++i)
          if (4 * i < live)
            rw_cp16(s + ((lane >> 3) + 4 * i) * kRwPitch + q * 4,
                    A + (off[i] < 0 ? 0 : (long long)off[i] * g.row_len + kc + q * 4), off[i] >= 0);
      }
      float* ws = s + kRwRows * kRwPitch;
      for (int e = lane * 4; e < kn * kNTile; e += 128) rw_cp16(ws + e, W + (long long)kc * kNTile + e, true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int rg = lane & 7, cg = lane >> 3;
  unsigned long long acc[kRwTR][4];
#pragma unroll
  for (int i = 0; i < kRwTR; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0ull;
  load(0, st);
  for (int kc = 0, b = 0; kc < K; kc += kRwKC, b ^= 1) {
    load(kc + kRwKC, st + (b ^ 1) * kRwStage);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    const float* As = st + b * kRwStage;
    const float* Ws = As + kRwRows * kRwPitch;
    const int kn = min(kRwKC, K - kc);
    if (live > 16)
      rw_stage<kRwTR>(As, Ws, kn, rg, cg, acc);
    else if (live > 8)
      rw_stage<2>(As, Ws, kn, rg, cg, acc);
    else
      rw_stage<1>(As, Ws, kn, rg, cg, acc);
    __syncwarp();  // every lane has read the stage before it is refilled
  }
  const int col = tile * kNTile + cg * 8;
  if (col >= g.n_cols) return;  // a multiple of 8
  float* P = static_cast<float*>(g.partial) + (long long)d * rows * g.n_cols;
#pragma unroll
  for (int i = 0; i < kRwTR; ++i) {
    const int r = r0 + rg + 8 * i;
    if (r >= rows) break;
    ulonglong2* o = reinterpret_cast<ulonglong2*>(P + (long long)r * g.n_cols + col);
    o[0] = make_ulonglong2(acc[i][0], acc[i][1]);
    o[1] = make_ulonglong2(acc[i][2], acc[i][3]);
  }
}

// C (+)= the levels' partial sums in neighbour order; a thread adds 4 values.
constexpr int kRwRed = 128;
__global__ void __launch_bounds__(kRwRed) nbr_rows_reduce_kernel(const __grid_constant__ RowsGroup G) {
  int i = 0;
  while (i + 1 < G.n && (int)blockIdx.x >= G.first[i + 1]) ++i;
  const NbrGemm& g = G.g[i];
  const long long count = (long long)g.grid[0] * g.grid[1] * g.grid[2] * g.n_cols;
  const long long e = ((long long)((int)blockIdx.x - G.first[i]) * kRwRed + threadIdx.x) * 4;
  if (e >= count) return;
  const float4* part = reinterpret_cast<const float4*>(static_cast<const float*>(g.partial) + e);
  float4* C = reinterpret_cast<float4*>(static_cast<float*>(g.C) + e);
  float4 s = g.accumulate ? *C : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 9
  for (int d = 0; d < 27; ++d) {
    if (d == 13 && g.skip_center) continue;
    const float4 v = __ldg(part + d * (count / 4));
    s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
  }
  *C = s;
}

}  // namespace

cudaError_t launch_nbr_gemm_rows(const NbrGemm* gs, int n, cudaStream_t s) {
  if (n < 1 || n > kRowsGroupMax) return cudaErrorInvalidValue;
  static SmemOptIn opt;
  if (cudaError_t e = opt(nbr_gemm_rows_kernel, kRwSmem)) return e;
  RowsGroup G{};
  long long per_tile = 0;
  for (int i = 0; i < n; ++i) {
    const long long rows = (long long)gs[i].grid[0] * gs[i].grid[1] * gs[i].grid[2];
    if (rows <= 0) continue;
    if (gs[i].ntiles != gs[0].ntiles || gs[i].dsplit != 27) return cudaErrorInvalidValue;
    G.g[G.n] = gs[i];
    G.first[G.n++] = (int)per_tile;
    per_tile += (rows + kRwRows - 1) / kRwRows * 27;
  }
  if (G.n == 0) return cudaSuccess;
  const long long items = per_tile * gs[0].ntiles;
  if (items > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  nbr_gemm_rows_kernel<<<(unsigned)items, 32, kRwSmem, s>>>(G, (int)per_tile);
  if (cudaError_t e = cudaGetLastError()) return e;
  long long blocks = 0;
  for (int i = 0; i < G.n; ++i) {
    const NbrGemm& g = G.g[i];
    G.first[i] = (int)blocks;
    blocks += ((long long)g.grid[0] * g.grid[1] * g.grid[2] * g.n_cols + kRwRed * 4 - 1) / (kRwRed * 4);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  }
  nbr_rows_reduce_kernel<<<(unsigned)blocks, kRwRed, 0, s>>>(G);
  return cudaGetLastError();
}

}  // namespace fmmgb
