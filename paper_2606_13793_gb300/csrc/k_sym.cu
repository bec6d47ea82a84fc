// Neighbour contractions on the CUDA cores in the reflection basis.
//
// The M2L of a level (Sec. 2.3, eq. M2L), the final-stage M2P (Sec. 4) and the
// near field of leaf-2 and leaf-4 boxes (eq. direct) are the contraction of k_gemm_simt.cu,
//   C[P][n] = sum_{d in 27 neighbours} sum_k A[P + d][k] W_d[k][n],
// and their weights are those of an even kernel: reflecting an axis about the
// target row's centre maps source position j (a child box, or a cell) to
// M - 1 - j (M positions per row and axis), target position t to M - 1 - t,
// and multiplies a component alpha / beta by its parity (-1)^alpha_q.  In the
// basis of sums and differences over the mirror pairs,
//   B+-[k] = A[M/2 + k] +- (-1)^alpha_q A[M/2 - 1 - k],   k = 0 .. 3M/2 - 1,
//   L+-[o] = L[M/2 + o] +- (-1)^beta_q  L[M/2 - 1 - o],   o = 0 .. M/2 - 1,
// per axis, the operator falls into 8 blocks (one per choice of the three
// signs) of 1/8 of the rows and 1/8 of the columns: 8 times fewer products,
// exactly, for ~3 additions per source value.  (M = 2: children of a parent,
// components alpha, or the cells of a leaf-2 box; M = 4: cells of a leaf-4
// box.  The M2P's targets are the 2 b cells of a parent per axis.)
//
// What bounds it: shared-memory reads and FMAs, about equally.  A source
// value takes 4 reads per (x, y) mirror pair and a weight serves the RZ rows
// of a thread, so per (component, x-y pair) a warp reads 10 RZ + 20 values
// and issues 6 RZ N FMAs and 13.5 RZ additions (M = 2, N = 8 columns).
//
// Forms:
//  * z-run (sym_m2l, sym_near4): a CTA covers 8 x 4 x RZ rows, lane = (x, y),
//    the RZ rows of a z-run in registers; warp = (sign of x, sign of y), both
//    signs of z in the two halves of a packed pair, so that the weights (one
//    pair per column) need no splat.  The four warps exchange their blocks
//    through shared memory at the end.  Against the direct z-run tiles of
//    k_gemm_zrun.cu (GB300): FP32 p = 6, 32^3 rows (256^3 cells) 1.48 -> 0.33
//    ms, its near field 1.11 -> 0.28 ms; FP64 p = 6, 12^3 rows 7.6 -> 1.1 ms,
//    24^3 boxes 2.9 -> 0.63 ms.  Of the issue slots ~45% are used: 8 warps an
//    SM, the 128 accumulator registers a thread (RZ = 8, N = 8) allow no more,
//    and shorter runs read more weights per product.
//  * rows (sym_rows, FP64): grids of few rows (the coarse levels): thread =
//    (component, row group) with all 8 blocks, one CTA per 16 (or 8) rows and
//    mirror triple k; partial sums of the 27 triples are added in order by
//    sym_reduce_kernel.  Levels that share a stream go in one launch (8 and 64
//    rows at p = 4: 0.62 -> 0.052 ms for both).
//  * tiny (sym_tiny): at most 64 rows inside a batch, without partial sums.
#include "fmm_internal.h"
#include "multi.cuh"

namespace fmmgb {
namespace {

constexpr int kSyThreads = 128;

__device__ __forceinline__ unsigned long long sy_fma2(unsigned long long a, unsigned long long b,
                                                      unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long sy_pack(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 sy_unpack(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Accumulators of one row and column, both signs of z (lo: +, hi: -).
template <typename T>
struct SyAcc;
template <>
struct SyAcc<float> {
  unsigned long long v = 0ull;
  __device__ __forceinline__ float lo() const { return sy_unpack(v).x; }
  __device__ __forceinline__ float hi() const { return sy_unpack(v).y; }
};
template <>
struct SyAcc<double> {
  double a = 0.0, b = 0.0;
  __device__ __forceinline__ double lo() const { return a; }
  __device__ __forceinline__ double hi() const { return b; }
};

// acc[r][n] += (u + f l) w+[n], (u - f l) w-[n] for the RZ rows and NL
// columns of one z mirror pair: u / l = v[r * M + uo] / v[r * M + lo].
template <int RZ, int NC, int NL, int M, int HV>
__device__ __forceinline__ void sy_step(const float (&v)[HV], int uo, int lo, float f, const float* w,
                                        SyAcc<float> (&acc)[RZ][NC]) {
  unsigned long long b[NL];
  if constexpr (NL % 2 == 0) {
#pragma unroll
    for (int n = 0; n < NL; n += 2) {
      const ulonglong2 q = reinterpret_cast<const ulonglong2*>(w)[n / 2];
      b[n] = q.x;
      b[n + 1] = q.y;
    }
  } else {
    b[0] = *reinterpret_cast<const unsigned long long*>(w);
  }
#pragma unroll
  for (int r = 0; r < RZ; ++r) {
    const float u = v[r * M + uo], l = v[r * M + lo];
    const unsigned long long a = sy_pack(fmaf(f, l, u), fmaf(-f, l, u));
#pragma unroll
    for (int n = 0; n < NL; ++n) acc[r][n].v = sy_fma2(a, b[n], acc[r][n].v);
  }
}
template <int RZ, int NC, int NL, int M, int HV>
__device__ __forceinline__ void sy_step(const double (&v)[HV], int uo, int lo, double f, const double* w,
                                        SyAcc<double> (&acc)[RZ][NC]) {
  double bp[RZ], bm[RZ];
#pragma unroll
  for (int r = 0; r < RZ; ++r) {
    const double u = v[r * M + uo], l = v[r * M + lo];
    bp[r] = fma(f, l, u);
    bm[r] = fma(-f, l, u);
  }
#pragma unroll
  for (int n = 0; n < NL; ++n) {
    const double2 q = reinterpret_cast<const double2*>(w)[n];
#pragma unroll
    for (int r = 0; r < RZ; ++r) {
      acc[r][n].a = fma(bp[r], q.x, acc[r][n].a);
      acc[r][n].b = fma(bm[r], q.y, acc[r][n].b);
    }
  }
}

// v[z] = (uu + fx lu) + fy (ul + fx ll): one (x, y) mirror pair of a halo
// column, z in 16-byte pieces.
template <int HV>
__device__ __forceinline__ void sy_column(float (&v)[HV], const float* uu, const float* lu, const float* ul,
                                          const float* ll, float fx, float fy) {
  static_assert(HV % 4 == 0, "whole 16-byte pieces");
  const unsigned long long fx2 = sy_pack(fx, fx), fy2 = sy_pack(fy, fy);
#pragma unroll
  for (int z = 0; z < HV; z += 4) {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(uu + z), b = *reinterpret_cast<const ulonglong2*>(lu + z);
    const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(ul + z), d = *reinterpret_cast<const ulonglong2*>(ll + z);
    const float2 p = sy_unpack(sy_fma2(fy2, sy_fma2(fx2, d.x, c.x), sy_fma2(fx2, b.x, a.x)));
    const float2 q = sy_unpack(sy_fma2(fy2, sy_fma2(fx2, d.y, c.y), sy_fma2(fx2, b.y, a.y)));
    v[z] = p.x, v[z + 1] = p.y, v[z + 2] = q.x, v[z + 3] = q.y;
  }
}
template <int HV>
__device__ __forceinline__ void sy_column(double (&v)[HV], const double* uu, const double* lu, const double* ul,
                                          const double* ll, double fx, double fy) {
#pragma unroll
  for (int z = 0; z < HV; z += 2) {
    const double2 a = *reinterpret_cast<const double2*>(uu + z), b = *reinterpret_cast<const double2*>(lu + z);
    const double2 c = *reinterpret_cast<const double2*>(ul + z), d = *reinterpret_cast<const double2*>(ll + z);
    v[z] = fma(fy, fma(fx, d.x, c.x), fma(fx, b.x, a.x));
    v[z + 1] = fma(fy, fma(fx, d.y, c.y), fma(fx, b.y, a.y));
  }
}

template <typename T>
__device__ __forceinline__ void cp_async_elt(T* dst, const T* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (sizeof(T) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Back from the reflection basis along the three bits of an 8-vector: bit q
// of the index is the sign (0: +) on entry and the side (1: upper) on exit;
// p: parity bits of the output component.
template <typename T>
__device__ __forceinline__ void sy_unfold(T (&v)[8], int p) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const T sg = (p >> q) & 1 ? T(-1) : T(1);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i & (1 << q)) continue;
      const T a = v[i], b = v[i | (1 << q)];
      v[i | (1 << q)] = a + b;
      v[i] = (a - b) * sg;
    }
  }
}

// ------------------------------------------------------------ M2L, z-run --

// A halo column's values lie along z, so a lane reads its z-run in 16-byte
// pieces; the pitch of a column keeps the 8 lanes of a quarter warp (adjacent
// columns) in different banks: a multiple of 16 bytes, 12 or 20 mod 32 words
// (or 4 or 28).
template <typename T>
constexpr int sy_pitch(int hv) {
  constexpr int V = 16 / (int)sizeof(T);  // values per 16 bytes
  int p = (hv + V - 1) / V * V;
  while ((p / V) % 2 == 0) p += V;  // an odd number of pieces
  return p;
}

// Halo of one component's child values: (8 + 2) x (4 + 2) x (RZ + 2) parents,
// stored [cx][jy][bx][jz].
constexpr int kMlStages = 3;
template <typename T, int RZ>
struct MlHalo {
  static constexpr int pz = sy_pitch<T>(2 * (RZ + 2));
  static constexpr int y = 10 * pz, x = 12 * y;  // strides of jy and of the child's x bit
  static constexpr int size = 2 * x;
};
constexpr int kMlW = 9 * 4 * 3 * 8 * 2;  // weights of one component: 9 (x, y) pairs, 8 columns
template <typename T, int RZ>
constexpr size_t sym_m2l_smem() {
  return sizeof(T) * (size_t)kMlStages * (MlHalo<T, RZ>::size + kMlW);
}

template <typename T, int RZ, int NL>
__device__ __forceinline__ void sy_ml_component(const T* raw, const T* W, int xy0, int nxy, int xl, int yl, T fx, T fy,
                                                T fz, bool skip0, SyAcc<T> (&acc)[RZ][8]) {
  constexpr int HV = 2 * (RZ + 2);
  for (int j = nxy - 1; j >= 0; --j) {  // far pairs first
    const int xy = xy0 + j, kx = xy % 3, ky = xy / 3;
    using H = MlHalo<T, RZ>;
    const int xu = ((3 + kx) & 1) * H::x + (xl + ((3 + kx) >> 1)) * H::pz;
    const int xlo = ((2 - kx) & 1) * H::x + (xl + ((2 - kx) >> 1)) * H::pz;
    const int yu = (2 * yl + 3 + ky) * H::y, ylo = (2 * yl + 2 - ky) * H::y;
    T v[HV];
    sy_column<HV>(v, raw + xu + yu, raw + xlo + yu, raw + xu + ylo, raw + xlo + ylo, fx, fy);
    const T* w = W + j * (4 * 3 * NL * 2);
#pragma unroll
    for (int kz = 2; kz >= 0; --kz) {
      if (kz == 0 && xy == 0 && skip0) continue;  // the own parent's block is zero
      sy_step<RZ, 8, NL, 2, HV>(v, 3 + kz, 2 - kz, fz, w + kz * NL * 2, acc);
    }
  }
}

template <typename T, int RZ>
__device__ __forceinline__ void sym_m2l_body(const NbrGemm& g, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sy_smem[];
  T* sm = reinterpret_cast<T*>(sy_smem);
  using H = MlHalo<T, RZ>;
  constexpr int kRaw = H::size, kStage = kRaw + kMlW;
  constexpr int kPos = (RZ + 2) * 60, kNp = (kPos + kSyThreads - 1) / kSyThreads;
  const SymTab& st = *g.st;
  const int u = (int)vb.y;
  if (u >= st.nunits) return;  // the launch has one block row per 32 columns, this form one per 64
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int xl = lane & 7, yl = lane >> 3;
  const int ntx = (g.grid[0] + 7) / 8, nty = (g.grid[1] + 3) / 4;
  const int bt = (int)vb.x;
  const int ox = (bt % ntx) * 8, oy = ((bt / ntx) % nty) * 4, oz = (bt / (ntx * nty)) * RZ;
  const int nxy = 9 / g.dsplit, xy0 = (g.dsplit > 1 ? (int)vb.z : 0) * nxy;
  const int n8 = st.n8[u], n4 = st.n4[u], K = st.n1[u];
  const T* A = static_cast<const T*>(g.A);
  const T* W = static_cast<const T*>(g.Ws) + st.w_off[u];

  int goff[kNp], soff[kNp];
#pragma unroll
  for (int i = 0; i < kNp; ++i) {
    const int e = t + i * kSyThreads;
    const int bx = e % 10, by = (e / 10) % 6, bz = e / 60;
    const int x = ox + bx - 1, y = oy + by - 1, z = oz + bz - 1;
    soff[i] = e < kPos ? by * 2 * H::y + bx * H::pz + bz * 2 : -1;
    goff[i] = (x >= 0 && y >= 0 && z >= 0 && x < g.grid[0] && y < g.grid[1] && z < g.grid[2])
                  ? (z * g.grid[1] + y) * g.grid[0] + x
                  : -1;
  }
  // Components from the highest order down: the low orders hold the bulk of a
  // sum, so its rounding is that of the last few additions.
  auto load = [&](int i) {
    const int a = K - 1 - i;
    if (a >= 0) {
      T* stg = sm + (i % kMlStages) * kStage;
      const T* Aa = A + (long long)a * 8 * g.lda;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        T* d = stg + (c >> 2) + ((c >> 1) & 1) * H::y + (c & 1) * H::x;
#pragma unroll
        for (int e = 0; e < kNp; ++e)
          if (soff[e] >= 0) cp_async_elt(d + soff[e], Aa + (goff[e] < 0 ? 0 : goff[e]), goff[e] >= 0);
        Aa += g.lda;
      }
      const int nl = a < n8 ? 8 : a < n4 ? 4 : 1;
      const long long wo = 216LL * (a < n8 ? 8 * a : a < n4 ? 8 * n8 + 4 * (a - n8) : 8 * n8 + 4 * (n4 - n8) + a - n4);
      const char* src = reinterpret_cast<const char*>(W + wo + xy0 * 24 * nl);
      char* dst = reinterpret_cast<char*>(stg + kRaw);
      const int bytes = nxy * 24 * nl * (int)sizeof(T);
      for (int e = t * 16; e < bytes; e += kSyThreads * 16) cp_async16(dst + e, src + e);
    }
    cp_async_commit();
  };

  SyAcc<T> acc[RZ][8];
  load(0);
  load(1);
  for (int i = 0; i < K; ++i) {
    cp_async_wait<1>();
    __syncthreads();  // the component has landed for every thread; the previous one's stage is free
    load(i + 2);
    const int a = K - 1 - i;
    const T* raw = sm + (i % kMlStages) * kStage;
    const int p = st.par[a];
    const T fx = ((p ^ warp) & 1) ? T(-1) : T(1), fy = (((p >> 1) ^ (warp >> 1)) & 1) ? T(-1) : T(1);
    const T fz = (p & 4) ? T(-1) : T(1);
    const int nl = a < n8 ? 8 : a < n4 ? 4 : 1;
    const T* w = raw + kRaw + warp * (6 * nl);
    if (nl == 8)
      sy_ml_component<T, RZ, 8>(raw, w, xy0, nxy, xl, yl, fx, fy, fz, g.skip_center, acc);
    else if (nl == 4)
      sy_ml_component<T, RZ, 4>(raw, w, xy0, nxy, xl, yl, fx, fy, fz, g.skip_center, acc);
    else
      sy_ml_component<T, RZ, 1>(raw, w, xy0, nxy, xl, yl, fx, fy, fz, g.skip_center, acc);
  }
  // Exchange the blocks (4 columns a pass) and write the children's values.
  const long long rows = (long long)g.grid[0] * g.grid[1] * g.grid[2];
  T* C = g.dsplit > 1 ? static_cast<T*>(g.partial) + (long long)vb.z * rows * g.n_cols : static_cast<T*>(g.C);
  const bool add = g.dsplit <= 1 && g.accumulate;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (u * 8 + h * 4 >= g.n_cols / 8) break;
    __syncthreads();  // the stages (first pass) or the previous pass's values are free
#pragma unroll
    for (int r = 0; r < RZ; ++r)
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        sm[((warp * RZ + r) * 4 + n) * 32 + lane] = acc[r][h * 4 + n].lo();
        sm[(((warp + 4) * RZ + r) * 4 + n) * 32 + lane] = acc[r][h * 4 + n].hi();
      }
    __syncthreads();
    const int be = u * 8 + h * 4 + warp;  // this warp's column
    const int x = ox + xl, y = oy + yl;
    if (be < g.n_cols / 8 && x < g.grid[0] && y < g.grid[1]) {
      const int p = g.sym == kSymM2p ? 0 : st.par[be];
#pragma unroll
      for (int r = 0; r < RZ; ++r) {
        const int z = oz + r;
        if (z >= g.grid[2]) break;
        T v[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) v[s] = sm[((s * RZ + r) * 4 + warp) * 32 + lane];
        sy_unfold(v, p);
        if (g.sym == kSymM2p) {  // cell `be` of the upper child, mirrored into the lower ones
          const int b = g.b, ox = be % b, oy = (be / b) % b, oz = be / (b * b);
          T* o = C + (((long long)z * g.grid[1] + y) * g.grid[0] + x) * g.n_cols;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int cx = (c & 1) ? ox : b - 1 - ox, cy = (c & 2) ? oy : b - 1 - oy, cz = (c & 4) ? oz : b - 1 - oz;
            T* oc = o + c * (b * b * b) + (cz * b + cy) * b + cx;
            *oc = add ? *oc + v[c] : v[c];
          }
          continue;
        }
        T* o = C + (((long long)z * g.grid[1] + y) * g.grid[0] + x) * g.n_cols + be * 8;
        if (add) {
#pragma unroll
          for (int c = 0; c < 8; ++c) v[c] += o[c];
        }
        constexpr int VN = 16 / (int)sizeof(T);
#pragma unroll
        for (int c = 0; c < 8; c += VN) *reinterpret_cast<uint4*>(o + c) = *reinterpret_cast<const uint4*>(&v[c]);
      }
    }
  }
}

template <typename T, int RZ>
__global__ void __launch_bounds__(kSyThreads, sizeof(T) == 4 ? (RZ <= 4 ? 3 : 2) : 1) sym_m2l_kernel(NbrGemm g) {
  sym_m2l_body<T, RZ>(g, native_vblock());
}

// ----------------------------------------------------- near field, leaf 4 --

// Halo of the density: (8 + 2) x (4 + 2) x (RZ + 2) boxes, stored
// [cx][jy][bx][jz] like the M2L's.
template <typename T, int RZ>
struct NfHalo {
  static constexpr int pz = sy_pitch<T>(4 * (RZ + 2));
  static constexpr int y = 10 * pz, x = 24 * y;
  static constexpr int size = 4 * x;
};
constexpr int kNfW = 36 * 4 * 6 * 8 * 2;
template <typename T>
constexpr bool kNfSmemW = sizeof(T) == 4;  // FP64: the weights stay in L1 / L2 (the DFMA pipe is the limit)
template <typename T, int RZ>
constexpr size_t sym_near4_smem() {
  return sizeof(T) * ((size_t)NfHalo<T, RZ>::size + (kNfSmemW<T> ? kNfW : 0));
}

template <typename T, int RZ>
__device__ __forceinline__ void sym_near4_body(const NbrGemm& g, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sy_smem[];
  using H = NfHalo<T, RZ>;
  T* raw = reinterpret_cast<T*>(sy_smem);
  if (vb.y) return;  // the launch has one block row per 32 columns; this form computes all 64 in one
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int xl = lane & 7, yl = lane >> 3;
  const int ntx = (g.grid[0] + 7) / 8, nty = (g.grid[1] + 3) / 4;
  const int bt = (int)vb.x;
  const int ox = (bt % ntx) * 8, oy = ((bt / ntx) % nty) * 4, oz = (bt / (ntx * nty)) * RZ;
  const int nxy = 36 / g.dsplit, xy0 = (g.dsplit > 1 ? (int)vb.z : 0) * nxy;
  const T* A = static_cast<const T*>(g.A);
  const T* W = static_cast<const T*>(g.Ws);
  if constexpr (kNfSmemW<T>) {
    T* Wsm = raw + H::size;
    const char* src = reinterpret_cast<const char*>(W + xy0 * 384);
    for (int i = t * 16; i < nxy * 384 * (int)sizeof(T); i += kSyThreads * 16)
      cp_async16(reinterpret_cast<char*>(Wsm) + i, src + i);
    cp_async_commit();
    W = Wsm;
  } else {
    W += xy0 * 384;
  }
  {
    // the halo's boxes: 16-byte pieces of box rows, lanes along x
    constexpr int VN = 16 / (int)sizeof(T), PB = 64 / VN;  // values a piece, pieces a box
    constexpr int kBoxes = 60 * (RZ + 2);
    for (int e = t; e < kBoxes; e += kSyThreads) {
      const int bx = e % 10, by = (e / 10) % 6, bz = e / 60;
      const int x = ox + bx - 1, y = oy + by - 1, z = oz + bz - 1;
      const bool in = x >= 0 && y >= 0 && z >= 0 && x < g.grid[0] && y < g.grid[1] && z < g.grid[2];
      const uint4* src =
          reinterpret_cast<const uint4*>(A + (in ? (((long long)z * g.grid[1] + y) * g.grid[0] + x) * 64 : 0));
      T* dst = raw + by * 4 * H::y + bx * H::pz + bz * 4;
#pragma unroll
      for (int q0 = 0; q0 < PB; q0 += 8) {
        uint4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = in ? __ldg(src + q0 + q) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const T* pv = reinterpret_cast<const T*>(&v[q]);
#pragma unroll
          for (int i = 0; i < VN; ++i) {
            const int cell = (q0 + q) * VN + i;  // x fastest
            dst[(cell >> 4) + (cell & 3) * H::x + ((cell >> 2) & 3) * H::y] = pv[i];
          }
        }
      }
    }
  }
  if constexpr (kNfSmemW<T>) cp_async_wait<0>();
  __syncthreads();

  const T fx = (warp & 1) ? T(-1) : T(1), fy = (warp & 2) ? T(-1) : T(1);
  constexpr int HV = 4 * (RZ + 2);
  SyAcc<T> acc[RZ][8];
  for (int j = nxy - 1; j >= 0; --j) {  // far pairs (small weights) first
    const int xy = xy0 + j, kx = xy % 6, ky = xy / 6;
    const int xu = ((2 + kx) & 3) * H::x + (xl + 1 + ((2 + kx) >> 2)) * H::pz;
    const int xlo = ((5 - kx) & 3) * H::x + (xl + ((5 - kx) >> 2)) * H::pz;
    const int yu = (4 * yl + 6 + ky) * H::y, ylo = (4 * yl + 5 - ky) * H::y;
    T v[HV];
    sy_column<HV>(v, raw + xu + yu, raw + xlo + yu, raw + xu + ylo, raw + xlo + ylo, fx, fy);
    const T* w = W + j * 384 + warp * 96;
#pragma unroll
    for (int kz = 5; kz >= 0; --kz) sy_step<RZ, 8, 8, 4, HV>(v, 6 + kz, 5 - kz, T(1), w + kz * 16, acc);
  }
  // Exchange the blocks, then one thread per box unfolds its 64 cells.
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RZ; ++r)
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      raw[((warp * 8 + n) * RZ + r) * 32 + lane] = acc[r][n].lo();
      raw[(((warp + 4) * 8 + n) * RZ + r) * 32 + lane] = acc[r][n].hi();
    }
  __syncthreads();
  const long long rows = (long long)g.grid[0] * g.grid[1] * g.grid[2];
  T* C = g.dsplit > 1 ? static_cast<T*>(g.partial) + (long long)vb.z * rows * g.n_cols : static_cast<T*>(g.C);
  const bool add = g.dsplit <= 1 && g.accumulate;
  const int x = ox + xl, y = oy + yl;
  if (x >= g.grid[0] || y >= g.grid[1]) return;
  for (int r = warp; r < RZ; r += 4) {
    const int z = oz + r;
    if (z >= g.grid[2]) break;
    T* o = C + (((long long)z * g.grid[1] + y) * g.grid[0] + x) * g.n_cols;
    T out[64];
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      T v[8];
#pragma unroll
      for (int s = 0; s < 8; ++s) v[s] = raw[((s * 8 + n) * RZ + r) * 32 + lane];
      sy_unfold(v, 0);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int tx = (c & 1) ? 2 + (n & 1) : 1 - (n & 1);
        const int ty = (c & 2) ? 2 + ((n >> 1) & 1) : 1 - ((n >> 1) & 1);
        const int tz = (c & 4) ? 2 + (n >> 2) : 1 - (n >> 2);
        out[(tz * 4 + ty) * 4 + tx] = v[c];
      }
    }
    if (add) {
#pragma unroll
      for (int c = 0; c < 64; ++c) out[c] += o[c];
    }
    constexpr int VN = 16 / (int)sizeof(T);
#pragma unroll
    for (int c = 0; c < 64; c += VN) *reinterpret_cast<uint4*>(o + c) = *reinterpret_cast<const uint4*>(&out[c]);
  }
}

template <typename T, int RZ>
__global__ void __launch_bounds__(kSyThreads, 1) sym_near4_kernel(NbrGemm g) {
  sym_near4_body<T, RZ>(g, native_vblock());
}

// ------------------------------------------------------------- M2L, rows --

// The 8 mirror positions of triple k = (kx, ky, kz) seen from one row.
struct SyTriple {
  int off[3][2];  // row offset of the upper / lower position per axis
  int cb[3][2];   // its child bit
  bool ok[3][2];  // inside the grid
  __device__ __forceinline__ SyTriple(const NbrGemm& g, int k, int rx, int ry, int rz) {
    const int kk[3] = {k % 3, (k / 3) % 3, k / 9};
    const int rr[3] = {rx, ry, rz}, str[3] = {1, g.grid[0], g.grid[0] * g.grid[1]};
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = h ? -kk[q] : 1 + kk[q];  // -2 .. 3
        const int d = j < 0 ? -1 : (j > 1 ? 1 : 0);
        cb[q][h] = j & 1;
        ok[q][h] = rr[q] + d >= 0 && rr[q] + d < g.grid[q];
        off[q][h] = d * str[q];
      }
  }
  // the row's 8 block values of one component (Aa: its child 0), parity p
  template <typename T>
  __device__ __forceinline__ void blocks(T (&v)[8], const T* Aa, long long lda, int row, bool live, int p) const {
#pragma unroll
    for (int m = 0; m < 8; ++m) {  // bit q: 0 upper, 1 lower along q
      const int hx = m & 1, hy = (m >> 1) & 1, hz = m >> 2;
      const int c = cb[0][hx] | (cb[1][hy] << 1) | (cb[2][hz] << 2);
      v[m] = (live && ok[0][hx] && ok[1][hy] && ok[2][hz])
                 ? __ldg(Aa + (long long)c * lda + row + off[0][hx] + off[1][hy] + off[2][hz])
                 : T(0);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const T f = (p >> q) & 1 ? T(-1) : T(1);
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        if (m & (1 << q)) continue;
        const T x = v[m], y = v[m | (1 << q)];
        v[m] = fma(f, y, x);
        v[m | (1 << q)] = fma(-f, y, x);
      }
    }
  }
};

// RC rows and the mirror triples [k0, k1) per CTA; thread = (component beta,
// group of RC / 8 rows), all 8 blocks in registers.  A triple's weights land
// by cp.async beside the staging loads, so the reduction loop reads shared
// memory only.
template <typename T, int RC>
constexpr size_t sym_rows_smem(int nk, int q_len) {
  return sizeof(T) * ((size_t)nk * 8 * RC + (size_t)q_len);
}

template <typename T, int RC>
__device__ __forceinline__ void sym_rows_body(const NbrGemm& g, int chunk, int k0, int k1) {
  extern __shared__ __align__(16) unsigned char sy_smem[];
  constexpr int R = RC / 8;
  const SymTab& st = *g.st;
  const int nk = st.nk;
  T* B = reinterpret_cast<T*>(sy_smem);  // [alpha][block][RC rows]
  T* Ws = B + nk * 8 * RC;               // one triple's weights: [alpha][beta][block]
  const int rows = g.grid[0] * g.grid[1] * g.grid[2];
  const int t = threadIdx.x, nt = blockDim.x;
  const T* A = static_cast<const T*>(g.A);
  const int be = t >> 3, rg = t & 7;
  // the warp's reach: its first column has the longest reduction
  const int bw = (t & ~31) >> 3;
  const int Kw = bw < nk ? st.kb[bw] : 0;
  T acc[8][R];
#pragma unroll
  for (int s = 0; s < 8; ++s)
#pragma unroll
    for (int i = 0; i < R; ++i) acc[s][i] = T(0);
  // staging: this thread's row (nt is a multiple of RC, so it is the same for all its components)
  const int sr = t % RC, row = chunk * RC + sr;
  const int rx = row % g.grid[0], ry = (row / g.grid[0]) % g.grid[1], rz = row / (g.grid[0] * g.grid[1]);
  for (int k = k0; k < k1; ++k) {
    if (k == 0 && g.skip_center) continue;
    const SyTriple tr(g, k, rx, ry, rz);
    __syncthreads();  // the previous triple's values are free
    {
      const char* src = reinterpret_cast<const char*>(static_cast<const T*>(g.Wq) + (long long)k * st.q_len);
      for (int i = t * 16; i < st.q_len * (int)sizeof(T); i += nt * 16)
        cp_async16(reinterpret_cast<char*>(Ws) + i, src + i);
      cp_async_commit();
    }
#pragma unroll 2
    for (int a = t / RC; a < nk; a += nt / RC) {
      T v[8];
      tr.blocks(v, A + (long long)a * 8 * g.lda, g.lda, row, row < rows, st.par[a]);
#pragma unroll
      for (int s = 0; s < 8; ++s) B[(a * 8 + s) * RC + sr] = v[s];
    }
    cp_async_wait<0>();
    __syncthreads();
    constexpr int VN = 16 / (int)sizeof(T);
#pragma unroll 2
    for (int a = Kw - 1; a >= 0; --a) {  // the low orders, the bulk of the sum, last
      T w[8];
      const uint4* wp = reinterpret_cast<const uint4*>(Ws + st.q_off[a] + be * 8);
#pragma unroll
      for (int s = 0; s < 8; s += VN) *reinterpret_cast<uint4*>(&w[s]) = wp[s / VN];
      const T* b = B + a * 8 * RC + rg * R;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        T x[R];
        if constexpr (R * sizeof(T) == 16) {
          *reinterpret_cast<uint4*>(x) = *reinterpret_cast<const uint4*>(b + s * RC);
        } else {
#pragma unroll
          for (int i = 0; i < R; ++i) x[i] = b[s * RC + i];
        }
#pragma unroll
        for (int i = 0; i < R; ++i) acc[s][i] = fma(x[i], w[s], acc[s][i]);
      }
    }
  }
  if (be >= nk) return;
  const int p = st.par[be];
  T* C = g.dsplit > 1 ? static_cast<T*>(g.partial) + (long long)k0 * rows * g.n_cols : static_cast<T*>(g.C);
  const bool add = g.dsplit <= 1 && g.accumulate;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int ro = chunk * RC + rg * R + i;
    if (ro >= rows) break;
    T v[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) v[s] = acc[s][i];
    sy_unfold(v, p);
    T* o = C + (long long)ro * g.n_cols + be * 8;
    if (add) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] += o[c];
    }
    constexpr int VN = 16 / (int)sizeof(T);
#pragma unroll
    for (int c = 0; c < 8; c += VN) *reinterpret_cast<uint4*>(o + c) = *reinterpret_cast<const uint4*>(&v[c]);
  }
}

// Several levels in one launch (blockIdx.y = triple where they are split):
// the coarse levels are independent and each alone is a few microseconds of
// latency, so together they cost about one.
struct SymGroup {
  NbrGemm g[kSymGroupMax];
  int first[kSymGroupMax + 1];  // first chunk (reduction: first block) of each level
  int n;
};

// Threads of a row-form block: 8 per component, orders up to p.
constexpr int sy_rows_threads(int p) { return ((p + 1) * (p + 1) * 8 + 31) / 32 * 32; }
template <typename T, int RC, int P>
__global__ void __launch_bounds__(sy_rows_threads(P)) sym_rows_kernel(const __grid_constant__ SymGroup G) {
  int i = 0;
  while (i + 1 < G.n && (int)blockIdx.x >= G.first[i + 1]) ++i;
  const int k0 = gridDim.y > 1 ? (int)blockIdx.y : 0;
  if (gridDim.y > 1 && k0 == 0 && G.g[i].skip_center) return;  // a zero triple, which the reduction leaves out
  sym_rows_body<T, RC>(G.g[i], (int)blockIdx.x - G.first[i], k0, gridDim.y > 1 ? k0 + 1 : 27);
}

// C (+)= the levels' partial sums, in order, compensated (the coarse levels
// carry the bulk of phi); a thread adds 16 bytes.
constexpr int kSyRedThreads = 128;
template <typename T>
__global__ void __launch_bounds__(kSyRedThreads) sym_reduce_kernel(const __grid_constant__ SymGroup G) {
  int i = 0;
  while (i + 1 < G.n && (int)blockIdx.x >= G.first[i + 1]) ++i;
  const NbrGemm& g = G.g[i];
  constexpr int VN = 16 / (int)sizeof(T);
  const long long count = (long long)g.grid[0] * g.grid[1] * g.grid[2] * g.n_cols;  // a multiple of 8
  const long long e = ((long long)((int)blockIdx.x - G.first[i]) * kSyRedThreads + threadIdx.x) * VN;
  if (e >= count) return;
  const T* part = static_cast<const T*>(g.partial) + e;
  T* C = static_cast<T*>(g.C) + e;
  T s[VN], lost[VN];  // the sum and what its additions rounded off
#pragma unroll
  for (int c = 0; c < VN; ++c) s[c] = g.accumulate ? C[c] : T(0), lost[c] = T(0);
#pragma unroll 9
  for (int d = 0; d < 27; ++d) {
    if (d == 0 && g.skip_center) continue;  // the own parent's triple is zero (nothing was written)
    T v[VN];
    *reinterpret_cast<uint4*>(v) = __ldg(reinterpret_cast<const uint4*>(part + d * count));
#pragma unroll
    for (int c = 0; c < VN; ++c) {  // two-sum: s + v = t + r exactly
      const T t = s[c] + v[c], b = t - s[c];
      lost[c] += (s[c] - (t - b)) + (v[c] - b);
      s[c] = t;
    }
  }
#pragma unroll
  for (int c = 0; c < VN; ++c) s[c] += lost[c];
  *reinterpret_cast<uint4*>(C) = *reinterpret_cast<const uint4*>(s);
}

// ------------------------------------------------- M2L, tiny grids (batch) --

// At most 64 rows, one block per 4 components beta, no partial sums (the
// batch's other blocks fill the GPU): four parts of 256 threads (row, beta)
// take every fourth triple, staging 8 components at a time, and are added in
// order at the end.
constexpr int kSyTinyParts = 4, kSyTinyThreads = 256 * kSyTinyParts, kSyTinyC = 8;
template <typename T>
constexpr size_t sym_tiny_smem() {
  return sizeof(T) * (size_t)kSyTinyParts * kSyTinyC * 8 * 64;
}

template <typename T>
__device__ __forceinline__ void sym_tiny_body(const NbrGemm& g, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sy_smem[];
  const SymTab& st = *g.st;
  const int part = threadIdx.x >> 8, tl = threadIdx.x & 255;
  T* all = reinterpret_cast<T*>(sy_smem);
  T* B = all + part * (kSyTinyC * 8 * 64);  // [component][block][64 rows]
  const int nk = st.nk, b0 = (int)vb.x * 4, be = b0 + (tl & 3), row = tl >> 2;
  const int rows = g.grid[0] * g.grid[1] * g.grid[2];
  const int K = b0 < nk ? st.kb[b0] : 0;
  const T* A = static_cast<const T*>(g.A);
  const int sr = tl & 63, rx = sr % g.grid[0], ry = (sr / g.grid[0]) % g.grid[1], rz = sr / (g.grid[0] * g.grid[1]);
  T acc[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) acc[s] = T(0);
  for (int a0 = (K - 1) / kSyTinyC * kSyTinyC; a0 >= 0; a0 -= kSyTinyC) {  // the low orders last
    for (int k0 = 0; k0 < 27; k0 += kSyTinyParts) {
      const int k = k0 + part;
      const bool on = k < 27 && !(k == 0 && g.skip_center);
      const T* W = static_cast<const T*>(g.Wq) + (long long)(on ? k : 0) * st.q_len + be * 8;
      __syncthreads();  // the previous components are read
      if (on) {
        const SyTriple tr(g, k, rx, ry, rz);
        for (int i = tl >> 6; i < kSyTinyC && a0 + i < K; i += 4) {
          T v[8];
          tr.blocks(v, A + (long long)(a0 + i) * 8 * g.lda, g.lda, sr, sr < rows, st.par[a0 + i]);
#pragma unroll
          for (int s = 0; s < 8; ++s) B[(i * 8 + s) * 64 + sr] = v[s];
        }
      }
      __syncthreads();
      if (on && row < rows)
        for (int i = min(kSyTinyC, K - a0) - 1; i >= 0; --i) {
          const T* w = W + st.q_off[a0 + i];
#pragma unroll
          for (int s = 0; s < 8; ++s) acc[s] = fma(B[(i * 8 + s) * 64 + row], __ldg(w + s), acc[s]);
        }
    }
  }
  __syncthreads();
  if (part > 0) {
#pragma unroll
    for (int s = 0; s < 8; ++s) B[s * 256 + tl] = acc[s];
  }
  __syncthreads();
  if (part > 0 || row >= rows || be >= nk) return;
#pragma unroll
  for (int q = 1; q < kSyTinyParts; ++q)
#pragma unroll
    for (int s = 0; s < 8; ++s) acc[s] += all[q * (kSyTinyC * 8 * 64) + s * 256 + tl];
  sy_unfold(acc, st.par[be]);
  T* o = static_cast<T*>(g.C) + (long long)row * g.n_cols + be * 8;
#pragma unroll
  for (int c = 0; c < 8; ++c) o[c] = g.accumulate ? o[c] + acc[c] : acc[c];
}

template <typename T>
__global__ void __launch_bounds__(kSyTinyThreads)
    sym_tiny_multi_kernel(const NbrGemm* __restrict__ gs, const MultiGrid* __restrict__ grids, int n, long long first) {
  __shared__ NbrGemm g;
  const long long b = (long long)blockIdx.x + first;
  const int i = multi_item_at(grids, n, b);
  if (threadIdx.x == 0) g = gs[i];
  __syncthreads();
  sym_tiny_body<T>(g, multi_vblock_at(grids[i], b));
}

// ---------------------------------------------------------- multi-item --

// Items of one launch: blocks [first, first + gridDim.x) of the step.
template <typename T, int RZ>
__global__ void __launch_bounds__(kSyThreads, sizeof(T) == 4 ? (RZ <= 4 ? 3 : 2) : 1)
    sym_m2l_multi_kernel(const NbrGemm* __restrict__ gs, const MultiGrid* __restrict__ grids, int n, long long first,
                         int ny) {
  __shared__ NbrGemm g;
  VBlock vb;
  const int i = multi_tile_major(grids, n, first, gridDim.x, ny, blockIdx.x, &vb);
  if (threadIdx.x == 0) g = gs[i];
  __syncthreads();
  sym_m2l_body<T, RZ>(g, vb);
}
template <typename T, int RZ>
__global__ void __launch_bounds__(kSyThreads, 1)
    sym_near4_multi_kernel(const NbrGemm* __restrict__ gs, const MultiGrid* __restrict__ grids, int n, long long first) {
  __shared__ NbrGemm g;
  const long long b = (long long)blockIdx.x + first;
  const int i = multi_item_at(grids, n, b);
  if (threadIdx.x == 0) g = gs[i];
  __syncthreads();
  sym_near4_body<T, RZ>(g, multi_vblock_at(grids[i], b));
}

template <typename T, int RZ>
cudaError_t launch_zrun_form(const NbrGemm& g, cudaStream_t s) {
  const long long tiles = (long long)((g.grid[0] + 7) / 8) * ((g.grid[1] + 3) / 4) * ((g.grid[2] + RZ - 1) / RZ);
  if (tiles <= 0) return cudaSuccess;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  if (g.sym == kSymNear4) {
    static SmemOptIn opt;
    if (cudaError_t e = opt(sym_near4_kernel<T, RZ>, sym_near4_smem<T, RZ>())) return e;
    sym_near4_kernel<T, RZ><<<dim3((unsigned)tiles, 1, (unsigned)g.dsplit), kSyThreads, sym_near4_smem<T, RZ>(), s>>>(g);
  } else {
    static SmemOptIn opt;
    if (cudaError_t e = opt(sym_m2l_kernel<T, RZ>, sym_m2l_smem<T, RZ>())) return e;
    sym_m2l_kernel<T, RZ><<<dim3((unsigned)tiles, (unsigned)((g.n_cols / 8 + 7) / 8), (unsigned)g.dsplit), kSyThreads,
                            sym_m2l_smem<T, RZ>(), s>>>(g);
  }
  return cudaGetLastError();
}

template <typename T, int RC, int P>
cudaError_t launch_rows_form(const NbrGemm* gs, int n, cudaStream_t s) {
  static SmemOptIn opt;
  if (cudaError_t e = opt(sym_rows_kernel<T, RC, P>, 227 * 1024)) return e;
  SymGroup G{};
  const int nk = gs[0].n_cols / 8, split = gs[0].dsplit;
  long long chunks = 0, blocks = 0;
  for (int i = 0; i < n; ++i) {
    const long long rows = (long long)gs[i].grid[0] * gs[i].grid[1] * gs[i].grid[2];
    if (rows <= 0) continue;
    G.g[G.n] = gs[i];
    G.first[G.n++] = (int)chunks;
    chunks += (rows + RC - 1) / RC;
    blocks += (rows * gs[i].n_cols * (long long)sizeof(T) + kSyRedThreads * 16 - 1) / (kSyRedThreads * 16);
    if (chunks > 0x7fffffffLL || blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  }
  if (G.n == 0) return cudaSuccess;
  const size_t smem = sym_rows_smem<T, RC>(nk, gs[0].q_len);
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  const int threads = (nk * 8 + 31) / 32 * 32;
  if (threads > sy_rows_threads(P)) return cudaErrorInvalidConfiguration;
  sym_rows_kernel<T, RC, P><<<dim3((unsigned)chunks, split > 1 ? 27u : 1u), threads, smem, s>>>(G);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || split <= 1) return e;
  blocks = 0;
  for (int i = 0; i < G.n; ++i) {
    const NbrGemm& g = G.g[i];
    G.first[i] = (int)blocks;
    blocks += ((long long)g.grid[0] * g.grid[1] * g.grid[2] * g.n_cols * (long long)sizeof(T) + kSyRedThreads * 16 - 1) /
              (kSyRedThreads * 16);
  }
  sym_reduce_kernel<T><<<(unsigned)blocks, kSyRedThreads, 0, s>>>(G);
  return cudaGetLastError();
}

template <typename T, int RZ>
cudaError_t launch_multi_form(int kind, const NbrGemm* gs, const MultiGrid* grids, int n, long long blocks,
                              long long first, int ny, cudaStream_t s) {
  if (kind == kSymNear4) {
    static SmemOptIn opt;
    if (cudaError_t e = opt(sym_near4_multi_kernel<T, RZ>, sym_near4_smem<T, RZ>())) return e;
    sym_near4_multi_kernel<T, RZ><<<(unsigned)blocks, kSyThreads, sym_near4_smem<T, RZ>(), s>>>(gs, grids, n, first);
  } else {
    static SmemOptIn opt;
    if (cudaError_t e = opt(sym_m2l_multi_kernel<T, RZ>, sym_m2l_smem<T, RZ>())) return e;
    sym_m2l_multi_kernel<T, RZ><<<(unsigned)blocks, kSyThreads, sym_m2l_smem<T, RZ>(), s>>>(gs, grids, n, first, ny);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_nbr_gemm_sym_rows(const NbrGemm* gs, int n, cudaStream_t s) {
  if (n < 1 || n > kSymGroupMax) return cudaErrorInvalidValue;
  for (int i = 0; i < n; ++i)
    if (gs[i].sym != kSymM2l || gs[i].shape != gs[0].shape || gs[i].dsplit != gs[0].dsplit || gs[i].st != gs[0].st)
      return cudaErrorInvalidValue;
  if (gs[0].n_cols > 8 * 49)  // order 7: fewer registers a thread
    return gs[0].shape == 0 ? launch_rows_form<double, 16, 8>(gs, n, s) : launch_rows_form<double, 8, 8>(gs, n, s);
  return gs[0].shape == 0 ? launch_rows_form<double, 16, 6>(gs, n, s) : launch_rows_form<double, 8, 6>(gs, n, s);
}

template <typename T>
cudaError_t launch_nbr_gemm_sym(const NbrGemm& g, cudaStream_t s) {
  constexpr bool f = sizeof(T) == 4;
  cudaError_t e;
  switch (g.shape) {
    case 0:
    case 3:  // the row form (FP64 only: FP32 levels of these shapes run direct)
      if constexpr (!f) return launch_nbr_gemm_sym_rows(&g, 1, s);
      return cudaErrorInvalidValue;
    case 1: e = launch_zrun_form<T, f ? 8 : 4>(g, s); break;
    case 2: e = launch_zrun_form<T, f ? 4 : 2>(g, s); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess || g.dsplit <= 1) return e;
  return launch_reduce_partials<T>(static_cast<const T*>(g.partial), g.dsplit,
                                   (long long)g.grid[0] * g.grid[1] * g.grid[2] * g.n_cols, static_cast<T*>(g.C),
                                   g.accumulate, s);
}

template <typename T>
cudaError_t launch_nbr_gemm_sym_multi(int shape, int kind, const NbrGemm* gs, const MultiGrid* grids, int n,
                                      long long blocks, long long first, int ny, cudaStream_t s) {
  constexpr bool f = sizeof(T) == 4;
  if (n <= 0 || blocks <= 0) return cudaSuccess;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  if (shape == 3) {
    if (kind != kSymM2l) return cudaErrorInvalidValue;
    static SmemOptIn opt;
    if (cudaError_t e = opt(sym_tiny_multi_kernel<T>, sym_tiny_smem<T>())) return e;
    sym_tiny_multi_kernel<T><<<(unsigned)blocks, kSyTinyThreads, sym_tiny_smem<T>(), s>>>(gs, grids, n, first);
    return cudaGetLastError();
  }
  return shape == 0   ? launch_multi_form<T, f ? 8 : 4>(kind, gs, grids, n, blocks, first, ny, s)
         : shape == 1 ? launch_multi_form<T, f ? 4 : 2>(kind, gs, grids, n, blocks, first, ny, s)
                      : launch_multi_form<T, f ? 6 : 3>(kind, gs, grids, n, blocks, first, ny, s);
}

template cudaError_t launch_nbr_gemm_sym<float>(const NbrGemm&, cudaStream_t);
template cudaError_t launch_nbr_gemm_sym<double>(const NbrGemm&, cudaStream_t);
template cudaError_t launch_nbr_gemm_sym_multi<float>(int, int, const NbrGemm*, const MultiGrid*, int, long long,
                                                      long long, int, cudaStream_t);
template cudaError_t launch_nbr_gemm_sym_multi<double>(int, int, const NbrGemm*, const MultiGrid*, int, long long,
                                                       long long, int, cudaStream_t);

}  // namespace fmmgb
