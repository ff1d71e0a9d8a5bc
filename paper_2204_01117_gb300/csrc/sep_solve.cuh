// Exact inverse of the finest-level pressure operator by separation of
// variables, the default preconditioner where its sizes allow (capi.cu,
// sep_available, use_sep).
//
// The operator of Sec. 3 has constant coefficients (buildings act through
// drag), so A = Tx + Ty + Tz with one tridiagonal matrix per axis: -1, 2, -1
// with 1 on the diagonal where the end is a wall or an inlet (dp/dn = 0) and
// 2 where it is an outlet (p = 0 in the ghost cell).  Ty and Tz are
// diagonalised by the cosines below (orthonormal rows phi_m, eigenvalues
// 4 sin^2(theta_m / 2)); what remains is one tridiagonal system along x per
// pair of modes.  z = A^-1 r is therefore
//   z transform, y transform, x solve, y transform back, z transform back
// (k_sep_init or k_sep_update, k_sep_y, k_sep_x, k_sep_y, k_sep_zi).  (Lynch, Rice and Thomas,
// "Direct solution of partial difference equations by tensor product
// methods", Numer. Math. 6, 1964.)
//
// In FP32 the inverse is exact to rounding, which leaves CG one or two
// iterations to 1e-7 where the V-cycle needs seven to eleven, and an
// application is 5 launches where the V-cycle has 14 to 18 that depend on
// one another.  CG still stops on ||r|| <= tol ||b|| with FP64 inner products,
// so the solution is the same to the same tolerance.  Its error against 64
// bits, over 3 to 9 seeds each of ten FP32 workloads (48 x 40 x 16 to 256 x 256 x
// 64, one to four steps), against the V-cycle's on the same inputs: u, v, w, k and
// omega 0.38 to 1.00 of it, p 0.77 to 1.10 (standard errors to 0.3: no difference
// that the seeds could tell).  Measured on a GB300, one time step with the V-cycle and
// with this in its first form, all else equal: 48 x 40 x 16 0.73 -> 0.20 ms, 157 x 203 x 41 1.87 -> 0.47 ms,
// 256 x 256 x 64 2.20 -> 1.09 ms, 512 x 768 x 1 1.24 -> 0.34 ms,
// 512 x 512 x 128 13.0 -> 8.7 ms (where the y transforms cost most); the
// longest axes that fit were all faster.
//
// The transforms are contractions of a field with a constant n x n matrix:
// tensor cores, TF32 operands split into a high and a low part (x = hi + lo,
// 11 bits each), three products hi hi + hi lo + lo hi accumulated in FP32.
// The dropped lo lo is at most 2^-22 of the product, the bit cut off either
// low part at most 2^-23: 2^-21 at worst where a plain FP32 product has 2^-24,
// which the errors above include.
//
// The modes of an axis with walls at both ends are even or odd about its
// middle, so there (always along z; along y for a wind along x) a transform
// takes the sums and the differences of mirrored cells through two matrices
// of half the size: half the products (a y transform
// of 512 x 512 x 128 0.61 -> 0.44 ms, of 256 x 256 x 64 47 -> 38 us; the
// solves need fewer iterations too, sums of half the length round less).
#pragma once
#include "mg_fused.cuh"

namespace uf {

constexpr int SEP_T = 256;        // threads of the transform kernels (8 warps)
constexpr int SEP_X_LINES = 8;    // lines (warps) per block of the x solve
constexpr int SEP_MAX_NX = 1024;  // 32 lanes x 32 values per line

// FP64 grids do the same on the FP64 pipe, 1/64 of the FP32 rate on this
// chip: the products are then what a pass costs, and a rule on the sizes
// keeps the V-cycle for the longest axes (sep_available in capi.cu, with both
// sides measured).
template <typename T>
struct SepMat { using type = float4; };   // FP32: see below
template <>
struct SepMat<double> { using type = double; };

// Separable solver of one grid.  FP32 matrices are packed in the order in
// which the lanes of a warp read the A operand of mma.m16n8k8: one float4 per
// lane and 16 x 8 tile, tiles row by row, zero beyond the matrix.  FP64
// matrices are stored column by column, each padded with zeros to an even
// number of rows.  A folded axis (SepAxis) has the matrix of its even modes,
// then that of its odd modes.
template <typename T>
struct Sep {
  using Mat = typename SepMat<T>::type;
  long long on;        // 0: this grid uses the V-cycle (8 bytes: no padding, the struct is compared bytewise)
  const Mat* yf;    // forward: row m = mode, column j = cell
  const Mat* yi;    // inverse (transpose)
  const Mat* zf;
  const Mat* zi;
  const T* piv;    // 1 / pivot of the x systems, one row of P per (y mode, z mode)
  T* t;                // scratch (padded cell arrays): z transforms and the y transform back write t,
  T* u;                // the y transform writes u, the x solve works on it in place
};

// Panel geometry.  The whole contracted axis of a set of columns of the field
// stays in shared memory.  FP32: a warp owns 32 rows x 32 columns of the
// result, a block (8 / WN) x WN warps; the row pitch of 8 mod 32 words gives
// the 32 lanes of a B fragment (4 rows x 8 columns) 32 banks.  FP64: panels of
// 32 columns (WN = 1); a warp owns 4 rows.
template <typename T, int WN>
constexpr int SEP_PITCH = sizeof(T) == 4 ? 32 * WN + 8 : 32;
// Columns of a y panel in units of 32: two while they fit with a full queue, else one.
constexpr int SEP_Y_WIDE = 688;
template <typename T>
__host__ __device__ inline int sep_y_wn(int ny) { return sizeof(T) == 4 && ny <= SEP_Y_WIDE ? 2 : 1; }
template <typename T>
constexpr int SEP_Z_WN = sizeof(T) == 4 ? 4 : 1;
// The axis of a transform: its cells (or modes) in one block of panel rows and
// one matrix, or folded in two, the even one of (n + 1) / 2 rows and the odd
// one of n / 2 rows, each padded with zero rows to a multiple of 8.
struct SepAxis {
  int n, fold;
  __host__ __device__ int size(int odd) const { return fold ? (n + 1 - odd) / 2 : odd ? 0 : n; }
  __host__ __device__ int pad(int odd) const { return (size(odd) + 7) / 8 * 8; }
  __host__ __device__ int rows() const { return pad(0) + pad(1); }
};
template <typename T>
__host__ __device__ inline size_t sep_block_count(int n) {   // elements of Sep<T>::Mat of an n x n matrix
  return sizeof(T) == 4 ? (size_t)((n + 15) / 16) * ((n + 7) / 8) * 32 : (size_t)n * ((n + 1) & ~1);
}
template <typename T>
__host__ __device__ inline size_t sep_mat_count(const SepAxis& x) { return sep_block_count<T>(x.size(0)) + sep_block_count<T>(x.size(1)); }
template <typename T>
__host__ __device__ inline SepAxis sep_axis_y(const Level<T>& L) { return {L.ny, !(L.out_mask & 12)}; }
template <typename T>
__host__ __device__ inline SepAxis sep_axis_z(const Level<T>& L) { return {L.nz, !(L.out_mask & 48)}; }
template <typename T>
__host__ __device__ inline size_t sep_panel_bytes(int wn, const SepAxis& x) {
  return sizeof(T) * (size_t)x.rows() * (sizeof(T) == 4 ? 32 * wn + 8 : 32);
}
// Behind an FP32 panel lies a queue of matrix tiles for each thread, four deep
// where a block's shared memory (227 KB) allows, else one.
constexpr int SEP_QUEUE = 4, SEP_SLOT = 2 * 16 * SEP_T;   // bytes of a slot: two tiles, 16 bytes per thread and tile
__host__ __device__ inline int sep_queue(int wn, const SepAxis& x) {
  return sep_panel_bytes<float>(wn, x) + SEP_QUEUE * SEP_SLOT + 1024 <= 227 * 1024 ? SEP_QUEUE : 1;
}
template <typename T>
__host__ __device__ inline size_t sep_smem(int wn, const SepAxis& x) {
  return sep_panel_bytes<T>(wn, x) + (sizeof(T) == 4 ? (size_t)sep_queue(wn, x) * SEP_SLOT : 0);
}
// Columns (x, y) of a z panel, and the blocks that cover the plane.  One cell
// in z has nothing to transform: the threads just share the columns out.
template <typename T>
__host__ __device__ inline int sep_z_cols(int nz) { return nz > 1 ? 32 * SEP_Z_WN<T> : (int)(16 / sizeof(T)) * SEP_T; }
template <typename T>
inline unsigned sep_z_blocks(int P, int ny, int nz) {
  return (unsigned)(((size_t)P * ny + sep_z_cols<T>(nz) - 1) / sep_z_cols<T>(nz));
}
// Blocks that share a y panel, each taking every split-th unit of result rows
// (sep_gemm).  Whole rounds of units while two blocks per SM have none, and
// single units where even one per SM would be idle otherwise: a quasi-2D or a
// small grid has fewer panels than SMs, and a warp's chain of products is what
// it waits for (512 x 768 x 1: 97 us unsplit, 37 by whole rounds, 31 by units;
// FP64 128 x 96 x 40: 152 and 120 us).
constexpr int SEP_SMS = 152;
template <typename T>
__host__ __device__ inline int sep_y_split(const Level<T>& L) {
  const SepAxis x = sep_axis_y(L);
  const int wn = sep_y_wn<T>(L.ny), unit = sizeof(T) == 4 ? 32 : 4, round = sizeof(T) == 4 ? 8 / wn : 8;
  const int units = (x.size(0) + unit - 1) / unit + (x.size(1) + unit - 1) / unit;
  const int panels = (L.P + 32 * wn - 1) / (32 * wn) * L.nz;
  const int resident = SEP_SMS * (sep_smem<T>(wn, x) <= 113 * 1024 ? 2 : 1);
  const int by_round = min((2 * SEP_SMS + panels - 1) / panels, (units + round - 1) / round);
  return max(by_round, min(resident / panels, units));
}

__device__ __forceinline__ void sep_put2(float* o, float a, float b) { *reinterpret_cast<float2*>(o) = make_float2(a, b); }
__device__ __forceinline__ void sep_put2(double* o, double a, double b) { *reinterpret_cast<double2*>(o) = make_double2(a, b); }
__device__ __forceinline__ float2 sep_get2(const float* o) { return *reinterpret_cast<const float2*>(o); }
__device__ __forceinline__ double2 sep_get2(const double* o) { return *reinterpret_cast<const double2*>(o); }
// A pointer into a cell array of the grid (UF_PTR).
#define SEP_PTR(p, base, L, width) UF_PTR(p, base, (L).P, (L).ny, (L).nz, width, BA_LEVEL)
// Results of a transform to rows of `pitch` values, `cols` columns of them.
template <typename T>
struct SepStore {
  T* __restrict__ dst;
  size_t pitch;
  long long cols;
  const Level<T>* L;   // (the array dst points into)
  const T* base;
  __device__ __forceinline__ int fetch(int, int) const { return 0; }
  __device__ __forceinline__ void operator()(int row, int col, T a, T b, int) const {
    if (col < cols) sep_put2(SEP_PTR(dst + row * pitch + col, base, *L, 2), a, b);
  }
};

// x = hi + lo (+ at most 2^-23 |x|): hi rounded to TF32's 11 bits, lo, of 12 at most, cut to them.
__device__ __forceinline__ void tf32_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  lo = __float_as_uint(__fsub_rn(x, __uint_as_float(hi))) & 0xffffe000u;
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void sep_copy16(void* to, const void* from, bool on) {   // zeros where not on
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "r"(on ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void sep_copy_tile(void* to, const void* from) {   // through L1: other warps want the same
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}
__device__ __forceinline__ void sep_copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void sep_copies_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The matrix tiles of a warp's work on their way to shared memory, `depth`
// ahead of its products: segment i (seg(i, a): the KT tiles behind each of a,
// 0 at the end), segment i + 1, ...  The first leave before the panel is
// loaded.  A thread copies the 16 bytes of each tile that its own MMAs read, so
// the queue needs no barrier; a slot is filled again once the products of its
// last content are issued.  (With one or two blocks of 8 warps per SM nothing
// else hides L2's latency: plain loads one tile ahead left the tensor pipe 43 %
// busy at n = 512, two ahead no more.  With the queue, the panel's copies all
// under way at once and the loads of r batched in the last transform: y of 512 x
// 512 x 128 443 -> 378 us, back along z 226 -> 151 us; 256 x 256 x 64 38 -> 34
// and 36 -> 27 us.)
template <int TILES, typename Seg>
struct SepQueue {
  float4* slots;
  const int depth;
  int slot = 0, i = 0, at = 0, KT;
  const float4* a[TILES];
  Seg seg;
  const float4* A;   // the axis' matrices
  const SepAxis x;
  __device__ __forceinline__ SepQueue(void* queue, int depth_, Seg seg_, const float4* A_, const SepAxis& x_)
      : slots(reinterpret_cast<float4*>(queue) + threadIdx.x), depth(depth_), seg(seg_), A(A_), x(x_) {
    KT = seg(0, a);
    for (int p = 0; p < depth; ++p) fill(p);
  }
  __device__ __forceinline__ void fill(int to) {
    if (at < KT) {
#pragma unroll
      for (int h = 0; h < TILES; ++h)
        sep_copy_tile(slots + to * (SEP_SLOT / 16) + h * SEP_T,
                      UF_PTR(a[h] + (size_t)at * 32, A, 32, 1, (long long)(sep_mat_count<float>(x) / 32), 1, BA_MATRIX));
      if (++at == KT) {
        at = 0;
        KT = seg(++i, a);
      }
    }
    sep_copies_commit();
  }
  // acc[h] += the next n tiles of row h times the 8 n panel rows at b.
  template <int WN>
  __device__ __forceinline__ void mma(float (&acc)[TILES][4][4], int n_tiles, const float* b) {
    constexpr int PB = SEP_PITCH<float, WN>;
#pragma unroll 2
    for (int kt = 0; kt < n_tiles; ++kt) {
      if (depth == SEP_QUEUE) sep_copies_wait<SEP_QUEUE - 1>();
      else sep_copies_wait<0>();
      uint32_t hi[TILES][4], lo[TILES][4];
#pragma unroll
      for (int h = 0; h < TILES; ++h) {
        const float4 c = slots[slot * (SEP_SLOT / 16) + h * SEP_T];
        tf32_split(c.x, hi[h][0], lo[h][0]);
        tf32_split(c.y, hi[h][1], lo[h][1]);
        tf32_split(c.z, hi[h][2], lo[h][2]);
        tf32_split(c.w, hi[h][3], lo[h][3]);
      }
      const float* bk = b + kt * 8 * PB;
      uint32_t bh[4][2], bl[4][2];
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        tf32_split(bk[n * 8], bh[n][0], bl[n][0]);
        tf32_split(bk[n * 8 + 4 * PB], bh[n][1], bl[n][1]);
      }
      // one product at a time over all accumulators: each waits for its own last product
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int h = 0; h < TILES; ++h) mma_tf32(acc[h][n], lo[h], bh[n][0], bh[n][1]);
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int h = 0; h < TILES; ++h) mma_tf32(acc[h][n], hi[h], bl[n][0], bl[n][1]);
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int h = 0; h < TILES; ++h) mma_tf32(acc[h][n], hi[h], bh[n][0], bh[n][1]);
      fill(slot);
      slot = slot + 1 == depth ? 0 : slot + 1;
    }
  }
};

// The transform of the block's panel sB ([rows][pitch], which panel() loads) by
// the matrices A of its axis, result rows in units of a warp: the block
// has units part, part + parts, ...  put(row, column of the panel
// (even), value, next value, what put.fetch(row, column) loaded).
//
// Forward, and both ways of an axis that is not folded: 32 rows a unit, those
// of the even modes first.
template <int WN, typename Panel, typename Put>
__device__ __forceinline__ void sep_gemm(const float4* __restrict__ A, const SepAxis& x, float* sB, int part, int parts,
                                         Panel panel, Put put) {
  constexpr int PB = SEP_PITCH<float, WN>, WM = 8 / WN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3, wm = warp / WN, wn = warp % WN;
  const int ue = (x.size(0) + 31) / 32, un = ue + (x.size(1) + 31) / 32;
  auto seg = [&](int i, const float4* (&a)[2]) {
    const int u = part + parts * (wm + WM * i);
    if (u >= un) return 0;
    const int odd = u >= ue, KT = x.pad(odd) / 8, m0 = 2 * (odd ? u - ue : u);
    const size_t tile = (size_t)m0 * KT + (odd ? (size_t)((x.size(0) + 15) / 16) * (x.pad(0) / 8) : 0);
    a[0] = A + tile * 32 + lane;
    a[1] = m0 * 16 + 16 < x.size(odd) ? a[0] + (size_t)KT * 32 : a[0];
    return KT;
  };
  SepQueue<2, decltype(seg)> queue(sB + x.rows() * PB, sep_queue(WN, x), seg, A, x);
  panel();
  __syncthreads();
  for (int u = part + parts * wm; u < un; u += WM * parts) {
    const int odd = u >= ue, M = x.size(odd), m0 = 2 * (odd ? u - ue : u);
    float acc[2][4][4] = {};
    queue.template mma<WN>(acc, x.pad(odd) / 8, sB + (t + (odd ? x.pad(0) : 0)) * PB + wn * 32 + g);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = (m0 + h) * 16 + g;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int col = wn * 32 + n * 8 + 2 * t;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int out = x.fold ? 2 * (row + 8 * q) + odd : row + 8 * q;
          if (row + 8 * q < M) put(out, col, acc[h][n][2 * q], acc[h][n][2 * q + 1], put.fetch(out, col));
        }
      }
    }
  }
}
// Back along a folded axis: 16 cells and their mirror images a unit, the even
// modes' sum plus and minus the odd ones'.
template <int WN, typename Panel, typename Put>
__device__ __forceinline__ void sep_gemm_back(const float4* __restrict__ A, const SepAxis& x, float* sB, int part, int parts,
                                              Panel panel, Put put) {
  if (!x.fold) return sep_gemm<WN>(A, x, sB, part, parts, panel, put);
  constexpr int PB = SEP_PITCH<float, WN>, WM = 8 / WN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3, wm = warp / WN, wn = warp % WN;
  const int Me = x.size(0), Mo = x.size(1), KE = x.pad(0) / 8, KO = x.pad(1) / 8;
  auto seg = [&](int i, const float4* (&a)[1]) {   // (only the last unit of all can lack odd modes)
    const int m = part + parts * (wm + WM * (i >> 1)), odd = i & 1;
    if (m * 16 >= x.size(odd)) return 0;
    a[0] = A + ((odd ? (size_t)((Me + 15) / 16) * KE : 0) + (size_t)m * (odd ? KO : KE)) * 32 + lane;
    return odd ? KO : KE;
  };
  SepQueue<1, decltype(seg)> queue(sB + x.rows() * PB, sep_queue(WN, x), seg, A, x);
  panel();
  __syncthreads();
  const float* b = sB + t * PB + wn * 32 + g;
  for (int m = part + parts * wm; m * 16 < Me; m += WM * parts) {
    float e[1][4][4] = {}, o[1][4][4] = {};
    queue.template mma<WN>(e, KE, b);
    if (m * 16 < Mo) queue.template mma<WN>(o, KO, b + x.pad(0) * PB);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = m * 16 + g + 8 * h, mirror = x.n - 1 - row;
      decltype(put.fetch(0, 0)) f[4][2] = {};   // what the results meet, all loads before the first use
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int col = wn * 32 + n * 8 + 2 * t;
        if (row < Me) f[n][0] = put.fetch(row, col);
        if (row < Mo) f[n][1] = put.fetch(mirror, col);
      }
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int col = wn * 32 + n * 8 + 2 * t;
        const float e0 = e[0][n][2 * h], e1 = e[0][n][2 * h + 1], o0 = o[0][n][2 * h], o1 = o[0][n][2 * h + 1];
        if (row < Me) put(row, col, e0 + o0, e1 + o1, f[n][0]);
        if (row < Mo) put(mirror, col, e0 - o0, e1 - o1, f[n][1]);
      }
    }
  }
}

// FP64: lane l owns columns 2 (l % 16), + 1 and rows 2 (l / 16), + 1 of its
// unit's four (A: column by column, an even number of rows each).
__device__ __forceinline__ void sep_fma(double (&c)[4], const double* __restrict__ A, int row, int M, const double* b) {
  const int MP = (M + 1) & ~1;
  const double* a = A + (row < M ? row : 0);
#pragma unroll 4
  for (int k = 0; k < M; ++k) {
    const double2 av = __ldg(reinterpret_cast<const double2*>(UF_PTR(a + (size_t)k * MP, A, MP, M, 1, 2, BA_MATRIX)));
    const double2 bv = *reinterpret_cast<const double2*>(b + k * 32);
    c[0] = fma(av.x, bv.x, c[0]);
    c[1] = fma(av.x, bv.y, c[1]);
    c[2] = fma(av.y, bv.x, c[2]);
    c[3] = fma(av.y, bv.y, c[3]);
  }
}
__device__ __forceinline__ size_t sep_mat64(int n) { return (size_t)n * ((n + 1) & ~1); }
template <int WN, typename Panel, typename Put>
__device__ __forceinline__ void sep_gemm(const double* __restrict__ A, const SepAxis& x, const double* sB, int part, int parts,
                                         Panel panel, Put put) {
  panel();
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = 2 * (lane & 15);
  const int ue = (x.size(0) + 3) / 4, un = ue + (x.size(1) + 3) / 4;
  for (int u = part + parts * warp; u < un; u += 8 * parts) {
    const int odd = u >= ue, M = x.size(odd), row = 4 * (odd ? u - ue : u) + 2 * (lane >> 4);
    double c[4] = {};
    sep_fma(c, A + (odd ? sep_mat64(x.size(0)) : 0), row, M, sB + (odd ? x.pad(0) * 32 : 0) + col);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int out = x.fold ? 2 * (row + h) + odd : row + h;
      if (row + h < M) put(out, col, c[2 * h], c[2 * h + 1], put.fetch(out, col));
    }
  }
}
template <int WN, typename Panel, typename Put>
__device__ __forceinline__ void sep_gemm_back(const double* __restrict__ A, const SepAxis& x, const double* sB, int part, int parts,
                                              Panel panel, Put put) {
  if (!x.fold) return sep_gemm<WN>(A, x, sB, part, parts, panel, put);
  panel();
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = 2 * (lane & 15);
  const int Me = x.size(0), Mo = x.size(1);
  for (int u = part + parts * warp; 4 * u < Me; u += 8 * parts) {
    const int row = 4 * u + 2 * (lane >> 4);
    double e[4] = {}, o[4] = {};
    sep_fma(e, A, row, Me, sB + col);
    if (row < Mo) sep_fma(o, A + sep_mat64(Me), row, Mo, sB + x.pad(0) * 32 + col);   // (no odd mode reaches the middle cell)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int mir = x.n - 1 - row - h;
      if (row + h < Me) put(row + h, col, e[2 * h] + o[2 * h], e[2 * h + 1] + o[2 * h + 1], put.fetch(row + h, col));
      if (row + h < Mo) put(mir, col, e[2 * h] - o[2 * h], e[2 * h + 1] - o[2 * h + 1], put.fetch(mir, col));
    }
  }
}

// The panel of a transform, 16 bytes a thread: columns col0 .., rows row0,
// row0 + step, ...  get(i) reads cell (or mode) i of the axis.  Forward, a
// folded axis stores the sums and then the differences of mirrored cells;
// back, its even modes and then its odd ones.
template <typename T, int PB, int UNROLL, typename Get>
__device__ __forceinline__ void sep_panel(T* sm, const SepAxis& x, int row0, int step, int col0, Get get) {
  using V = Vec16<T>;
  const int pe = x.pad(0), po = x.pad(1);
#pragma unroll UNROLL
  for (int k = row0; k < pe; k += step) {
    V a = {}, b = {};
    if (k < x.size(0)) a = get(k);
    if (k < x.size(1)) {
      b = get(x.n - 1 - k);
#pragma unroll
      for (int e = 0; e < V::N; ++e) {
        const T s = a.e[e] + b.e[e], d = a.e[e] - b.e[e];
        a.e[e] = s;
        b.e[e] = d;
      }
    }
    *reinterpret_cast<V*>(sm + k * PB + col0) = a;
    if (k < po) *reinterpret_cast<V*>(sm + (pe + k) * PB + col0) = b;
  }
}
// (Back: asynchronous copies, all rows under way at once; mode i of the
// thread's columns lies at from + i pitch, and counts where `in`.)
template <typename T, int PB>
__device__ __forceinline__ void sep_panel_back(T* sm, const SepAxis& x, int row0, int step, int col0, const T* from, size_t pitch,
                                               bool in, const Level<T>& L, const T* base) {
  const int pe = x.pad(0), rows = x.rows();
#pragma unroll 2
  for (int k = row0; k < rows; k += step) {
    const int odd = k >= pe, m = odd ? k - pe : k;
    const bool on = in && m < x.size(odd);
    sep_copy16(sm + k * PB + col0, SEP_PTR(from + (on ? (size_t)(x.fold ? 2 * m + odd : m) * pitch : 0), base, L, Vec16<T>::N), on);
  }
  sep_copies_commit();
  sep_copies_wait<0>();
}

// ------------------------------------------------------- z transforms ----
// A panel is 128 consecutive columns (x, y) of the P x ny plane with every z
// in shared memory, so each cell is read once; what the panel holds is formed
// while it is loaded: the first residual before the CG loop (sep_init_body),
// the CG update inside it (sep_update_body), with ||r||^2 and the convergence
// test.  Columns in the row padding (x >= nx) are zero.
template <typename T>
struct SepCols {   // a thread's 16 bytes of every row it loads
  bool flat;       // one cell in z: the identity, a thread per 16 bytes
  int row0, col0;
  size_t PS, c;    // cells of a plane, the first column
  bool in;
  int left_x;      // how many of the values lie inside the domain
  static constexpr int VR = 32 * SEP_Z_WN<T> / Vec16<T>::N;
  __device__ __forceinline__ SepCols(const Level<T>& L, const VBlock& vb) {
    static_assert(SEP_T % VR == 0, "a thread keeps its columns");
    flat = L.nz == 1;
    row0 = flat ? 0 : threadIdx.x / VR;
    col0 = Vec16<T>::N * (flat ? threadIdx.x : threadIdx.x % VR);
    PS = (size_t)L.P * L.ny;
    c = (size_t)vb.x * sep_z_cols<T>(L.nz) + col0;
    in = c < PS;
    left_x = L.nx - (int)(c % L.P);
  }
};
// t = Qz (what get gives: 16 bytes of plane k).
template <int UNROLL, typename T, typename Get>
__device__ __forceinline__ void sep_zf(const Level<T>& L, const Sep<T>& S, const SepCols<T>& C, const VBlock& vb, Get get) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  using V = Vec16<T>;
  constexpr int WN = SEP_Z_WN<T>, PB = SEP_PITCH<T, WN>;
  if (C.flat) {
    const V v = get(0);
    if (C.in) *reinterpret_cast<V*>(SEP_PTR(S.t + C.c, S.t, L, V::N)) = v;
    return;
  }
  const SepAxis ax = sep_axis_z(L);
  auto panel = [&] { sep_panel<T, PB, UNROLL>(sep_sm, ax, C.row0, SEP_T / C.VR, C.col0, get); };
  const size_t cb = (size_t)vb.x * 32 * WN;
  sep_gemm<WN>(S.zf, ax, sep_sm, 0, 1, panel, SepStore<T>{S.t + cb, C.PS, (long long)(C.PS - cb), &L, S.t});
}

__device__ __forceinline__ float sep_diff(float2 a, float2 b) { return ps_diff(a, b); }
__device__ __forceinline__ float sep_diff(float a, float b) { return a - b; }
__device__ __forceinline__ double sep_diff(double a, double b) { return a - b; }
__device__ __forceinline__ float sep_value(float2 a) { return ps_value(a); }
__device__ __forceinline__ float sep_value(float a) { return a; }
__device__ __forceinline__ double sep_value(double a) { return a; }
// A f (level_apply) at 16 bytes' worth of cells of plane k; f holds values or
// the pressure store's pairs, whose differences are taken on the pairs.
template <typename E, typename T>
__device__ __forceinline__ Vec16<T> sep_apply(const Level<T>& L, const SepCols<T>& C, const E* __restrict__ f, int k) {
  constexpr int N = Vec16<T>::N;
  struct alignas(16) Row { E e[N]; };
  const int i0 = L.nx - C.left_x, j = (int)(C.c / L.P);
  [[maybe_unused]] const E* __restrict__ f0 = f;   // (SEP_PTR)
  f += (size_t)k * C.PS + C.c;
  auto row = [&](const E* at) { return *reinterpret_cast<const Row*>(SEP_PTR(at, f0, L, N)); };
  const bool y0 = j > 0, y1 = j < L.ny - 1, z0 = k > 0, z1 = k < L.nz - 1;
  const Row m = row(f);
  Row ym = m, yp = m, zm = m, zp = m;
  E xm = m.e[0], xp = m.e[N - 1];
  if (y0) ym = row(f - L.P);
  if (y1) yp = row(f + L.P);
  if (z0) zm = row(f - C.PS);
  if (z1) zp = row(f + C.PS);
  if (i0 > 0) xm = *SEP_PTR(f - 1, f0, L, 1);
  if (C.left_x > N) xp = *SEP_PTR(f + N, f0, L, 1);
  Vec16<T> a;
#pragma unroll
  for (int e = 0; e < N; ++e) {
    const T v = (T)sep_value(m.e[e]);
    T s = 0;
    if (e > 0 || i0 > 0) s += L.wx * (T)sep_diff(m.e[e], e > 0 ? m.e[e - 1] : xm); else if (L.out_mask & 1) s += L.wx * v;
    if (e < C.left_x - 1) s += L.wx * (T)sep_diff(m.e[e], e < N - 1 ? m.e[e + 1] : xp); else if (L.out_mask & 2) s += L.wx * v;
    if (y0) s += L.wy * (T)sep_diff(m.e[e], ym.e[e]); else if (L.out_mask & 4) s += L.wy * v;
    if (y1) s += L.wy * (T)sep_diff(m.e[e], yp.e[e]); else if (L.out_mask & 8) s += L.wy * v;
    if (z0) s += L.wz * (T)sep_diff(m.e[e], zm.e[e]); else if (L.out_mask & 16) s += L.wz * v;
    if (z1) s += L.wz * (T)sep_diff(m.e[e], zp.e[e]); else if (L.out_mask & 32) s += L.wz * v;
    a.e[e] = s;
  }
  return a;
}

// Set-up of the solve: what k_cg_init does for the V-cycle (r = b - A g and a
// correction x from zero, or r = b - A x), and its z transform, in one pass
// (256 x 256 x 64: 68 us for the two kernels, 49 for this; 512 x 512 x 128: 345
// and 307).
template <typename T>
__device__ __forceinline__ void sep_init_body(const Level<T>& L, const Sep<T>& S, const T* __restrict__ b, T* __restrict__ x,
                                              const PStore<T>* __restrict__ g, double* partials, SolveState* st,
                                              cudaGraphConditionalHandle cond, int use_cond, int* left, const VBlock& vb) {
  __shared__ double sh[32];
  __shared__ bool last;
  using V = Vec16<T>;
  const SepCols<T> C(L, vb);
  const bool zero_rhs = st->bb == 0.0;
  DotAcc<T> dacc;
  sep_zf<1>(L, S, C, vb, [&](int k) {
    V v = {};
    if (!C.in) return v;
    const size_t o = (size_t)k * C.PS + C.c;
    if (!zero_rhs) {
      const V bv = *reinterpret_cast<const V*>(SEP_PTR(b + o, b, L, V::N));
      const V a = g ? sep_apply(L, C, g, k) : sep_apply(L, C, (const T*)x, k);
#pragma unroll
      for (int e = 0; e < V::N; ++e) {
        v.e[e] = e < C.left_x ? bv.e[e] - a.e[e] : T(0);
        dacc.add(v.e[e], v.e[e]);
      }
    }
    if (zero_rhs || g) *reinterpret_cast<V*>(SEP_PTR(x + o, x, L, V::N)) = V{};
    *reinterpret_cast<V*>(SEP_PTR(L.r + o, L.r, L, V::N)) = v;
    return v;
  });
  const double vals[1] = {block_sum<SEP_T>(dacc.value(), sh)};
  if (publish_partials<1>(partials, &st->ticket[1], vals, &last, vb)) {
    double tot[1];
    reduce_partials_sum<SEP_T, 1>(partials, tot, sh, vb.n);
    if (threadIdx.x == 0) {
      finish_init(st, tot[0], zero_rhs, cond, use_cond, left);
      st->ticket[1] = 0u;
    }
  }
}

// CG update x += alpha d, r -= alpha q and the z transform of the new r.
template <typename T>
__device__ __forceinline__ void sep_update_body(const Level<T>& L, const Sep<T>& S, T* __restrict__ x, const T* d0, const T* d1,
                                                const T* __restrict__ q, double* partials, SolveState* st,
                                                cudaGraphConditionalHandle cond, int use_cond, int* left, const VBlock& vb) {
  __shared__ double sh[32];
  __shared__ bool last;
  if (st->converged) return;
  using V = Vec16<T>;
  const SepCols<T> C(L, vb);
  const int it0 = st->iter;
  const T alpha = (T)st->alpha;
  const T* dn = (it0 & 1) ? d0 : d1;
  DotAcc<T> dacc;
  sep_zf<2>(L, S, C, vb, [&](int k) {
    V v = {};
    if (!C.in) return v;
    const size_t o = (size_t)k * C.PS + C.c;
    v = *reinterpret_cast<const V*>(SEP_PTR(L.r + o, L.r, L, V::N));
    const V qv = *reinterpret_cast<const V*>(SEP_PTR(q + o, q, L, V::N));
    const V dv = *reinterpret_cast<const V*>(SEP_PTR(dn + o, dn, L, V::N));
    V xv = *reinterpret_cast<const V*>(SEP_PTR(x + o, x, L, V::N));
#pragma unroll
    for (int e = 0; e < V::N; ++e) {
      v.e[e] = e < C.left_x ? v.e[e] - alpha * qv.e[e] : T(0);
      xv.e[e] = e < C.left_x ? xv.e[e] + alpha * dv.e[e] : T(0);
      dacc.add(v.e[e], v.e[e]);
    }
    *reinterpret_cast<V*>(SEP_PTR(L.r + o, L.r, L, V::N)) = v;
    *reinterpret_cast<V*>(SEP_PTR(x + o, x, L, V::N)) = xv;
    return v;
  });
  const double vals[1] = {block_sum<SEP_T>(dacc.value(), sh)};
  if (publish_partials<1>(partials, &st->ticket[3], vals, &last, vb)) {
    double tot[1];
    reduce_partials_sum<SEP_T, 1>(partials, tot, sh, vb.n);
    if (threadIdx.x == 0) {
      finish_rr(st, tot[0], it0, cond, use_cond, left);
      st->ticket[3] = 0u;
    }
  }
}

// z and the terms of r.z (rows of `pitch` values, `cols` columns of them).
template <typename T>
struct SepStoreDot {
  const T* __restrict__ r;
  T* __restrict__ z;
  size_t pitch;
  long long cols;
  DotAcc<T>* dot;
  const Level<T>* L;   // (the arrays r and z point into)
  const T *r0, *z0;
  using Pair = decltype(sep_get2((const T*)nullptr));
  __device__ __forceinline__ Pair fetch(int row, int col) const { return col < cols ? sep_get2(SEP_PTR(r + row * pitch + col, r0, *L, 2)) : Pair{}; }
  __device__ __forceinline__ void operator()(int row, int col, T a, T b, Pair rv) const {
    if (col >= cols) return;
    sep_put2(SEP_PTR(z + row * pitch + col, z0, *L, 2), a, b);
    dot->add(rv.x, a);
    dot->add(rv.y, b);
  }
};
// Back along z: z = Qz^T t, and r.z (from the first iteration on also beta).
template <typename T>
__device__ __forceinline__ void sep_zi_body(const Level<T>& L, const Sep<T>& S, T* __restrict__ z, double* partials, SolveState* st,
                                            const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  __shared__ double sh[32];
  __shared__ bool last;
  if (st->converged) return;
  using V = Vec16<T>;
  constexpr int WN = SEP_Z_WN<T>, BN = 32 * WN, PB = SEP_PITCH<T, WN>, VR = BN / V::N;
  const size_t PS = (size_t)L.P * L.ny;
  const bool flat = L.nz == 1;
  const int col0 = V::N * (flat ? threadIdx.x : threadIdx.x % VR);
  const size_t c = (size_t)vb.x * sep_z_cols<T>(L.nz) + col0;
  DotAcc<T> dacc;
  if (flat) {
    if (c < PS) {
      const V v = *reinterpret_cast<const V*>(SEP_PTR(S.t + c, S.t, L, V::N));
      const SepStoreDot<T> put{L.r + c, z + c, PS, V::N, &dacc, &L, L.r, z};
#pragma unroll
      for (int e = 0; e < V::N; e += 2) put(0, e, v.e[e], v.e[e + 1], put.fetch(0, e));
    }
  } else {
    const SepAxis ax = sep_axis_z(L);
    auto panel = [&] { sep_panel_back<T, PB>(sep_sm, ax, threadIdx.x / VR, SEP_T / VR, col0, S.t + (c < PS ? c : 0), PS, c < PS, L, S.t); };
    const size_t cb = (size_t)vb.x * BN;
    sep_gemm_back<WN>(S.zi, ax, sep_sm, 0, 1, panel, SepStoreDot<T>{L.r + cb, z + cb, PS, (long long)(PS - cb), &dacc, &L, L.r, z});
  }
  const double vals[1] = {block_sum<SEP_T>(dacc.value(), sh)};
  if (publish_partials<1>(partials, &st->ticket[0], vals, &last, vb)) {
    double tot[1];
    reduce_partials_sum<SEP_T, 1>(partials, tot, sh, vb.n);
    if (threadIdx.x == 0) {
      finish_rz(st, tot[0], st->iter > 0);
      st->ticket[0] = 0u;
    }
  }
}

// --------------------------------------------------------- y transforms --
// One panel of 32 WN columns of a z plane, every y; blocks vb.y of `split`
// share the panel's result rows.
template <int WN, bool INVERSE, typename T>
__device__ __forceinline__ void sep_y_panel(const Level<T>& L, const Sep<T>& S, int split, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  using V = Vec16<T>;
  constexpr int BN = 32 * WN, PB = SEP_PITCH<T, WN>, VR = BN / V::N;
  const SepAxis ax = sep_axis_y(L);
  const int x0 = vb.x * BN, xv = V::N * (threadIdx.x % VR), row0 = threadIdx.x / VR;
  const size_t base = (size_t)vb.z * L.P * L.ny + x0;
  const bool in = x0 + xv < L.P;
  const T* __restrict__ from = INVERSE ? S.u : S.t;
  T* __restrict__ to = INVERSE ? S.t : S.u;
  const T* __restrict__ src = from + base;
  T* __restrict__ dst = to + base;
  auto get = [&](int j) {
    V v = {};
    if (in) v = *reinterpret_cast<const V*>(SEP_PTR(src + (size_t)j * L.P + xv, from, L, V::N));
    return v;
  };
  const SepStore<T> put{dst, (size_t)L.P, L.P - x0, &L, to};
  if (INVERSE) {
    auto panel = [&] { sep_panel_back<T, PB>(sep_sm, ax, row0, SEP_T / VR, xv, src + (in ? xv : 0), (size_t)L.P, in, L, from); };
    sep_gemm_back<WN>(S.yi, ax, sep_sm, vb.y, split, panel, put);
  } else {
    auto panel = [&] { sep_panel<T, PB, 4>(sep_sm, ax, row0, SEP_T / VR, xv, get); };
    sep_gemm<WN>(S.yf, ax, sep_sm, vb.y, split, panel, put);
  }
}
template <bool INVERSE, typename T>
__device__ __forceinline__ void sep_y_body(const Level<T>& L, const Sep<T>& S, const SolveState* st, const VBlock& vb) {
  if (st->converged) return;
  const int split = sep_y_split(L);
  if (sizeof(T) == 4 && L.ny <= SEP_Y_WIDE) sep_y_panel<sizeof(T) == 4 ? 2 : 1, INVERSE>(L, S, split, vb);
  else sep_y_panel<1, INVERSE>(L, S, split, vb);
}

// -------------------------------------------------------------- x solve --
// One warp per line (a row of the padded array): forward y_i = f_i + e_{i-1}
// y_{i-1}, backward x_i = e_i (y_i + x_{i+1}) with e the reciprocal pivots of
// the line's tridiagonal matrix.  Lane l holds E consecutive values; each
// recurrence is a scan of the affine maps of the lanes (Blelloch 1990), so a
// line takes 10 shuffle steps instead of 2 nx dependent ones.  In the row
// padding e = 0, which makes the solution 0 there.
template <int E, typename T>
__device__ __forceinline__ void sep_x_line(T* __restrict__ row, const T* __restrict__ piv, int P) {
  using V = Vec16<T>;
  const int lane = threadIdx.x & 31;
  T f[E], e[E];
  if (E >= V::N) {
#pragma unroll
    for (int m = 0; m < E; m += V::N) {
      const int i = lane * E + m;
      V a = {}, b = {};
      if (i < P) {
        a = *reinterpret_cast<const V*>(row + i);
        b = *reinterpret_cast<const V*>(piv + i);
      }
#pragma unroll
      for (int q = 0; q < V::N && m + q < E; ++q) {
        f[m + q] = a.e[q];
        e[m + q] = b.e[q];
      }
    }
  } else {
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int i = lane * E + m;
      f[m] = i < P ? row[i] : T(0);
      e[m] = i < P ? piv[i] : T(0);
    }
  }
  // forward
  T ep = __shfl_up_sync(0xffffffffu, e[E - 1], 1);
  if (lane == 0) ep = T(0);
  T a = ep, b = f[0];   // the lane's map: last y = a * (y of the lane before) + b
#pragma unroll
  for (int m = 1; m < E; ++m) {
    b = fma(e[m - 1], b, f[m]);
    a *= e[m - 1];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T a2 = __shfl_up_sync(0xffffffffu, a, o), b2 = __shfl_up_sync(0xffffffffu, b, o);
    if (lane >= o) {
      b = fma(a, b2, b);
      a *= a2;
    }
  }
  T cin = __shfl_up_sync(0xffffffffu, b, 1);
  if (lane == 0) cin = T(0);
  f[0] = fma(ep, cin, f[0]);
#pragma unroll
  for (int m = 1; m < E; ++m) f[m] = fma(e[m - 1], f[m - 1], f[m]);
  // backward
  a = T(1);
  b = T(0);
#pragma unroll
  for (int m = E - 1; m >= 0; --m) {
    b = e[m] * (f[m] + b);
    a *= e[m];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T a2 = __shfl_down_sync(0xffffffffu, a, o), b2 = __shfl_down_sync(0xffffffffu, b, o);
    if (lane + o < 32) {
      b = fma(a, b2, b);
      a *= a2;
    }
  }
  cin = __shfl_down_sync(0xffffffffu, b, 1);
  if (lane == 31) cin = T(0);
#pragma unroll
  for (int m = E - 1; m >= 0; --m) cin = f[m] = e[m] * (f[m] + cin);
  if (E >= V::N) {
#pragma unroll
    for (int m = 0; m < E; m += V::N) {
      const int i = lane * E + m;
      V a;
#pragma unroll
      for (int q = 0; q < V::N && m + q < E; ++q) a.e[q] = f[m + q];
      if (i < P) *reinterpret_cast<V*>(row + i) = a;
    }
  } else {
#pragma unroll
    for (int m = 0; m < E; ++m)
      if (lane * E + m < P) row[lane * E + m] = f[m];
  }
}
template <typename T>
__device__ __forceinline__ void sep_x_body(const Level<T>& L, const Sep<T>& S, const SolveState* st, const VBlock& vb) {
  if (st->converged) return;
  const int line = vb.x * SEP_X_LINES + (threadIdx.x >> 5);
  if (line >= L.ny * L.nz) return;
  T* row = SEP_PTR(S.u + (size_t)line * L.P, S.u, L, L.P);
  const T* piv = SEP_PTR(S.piv + (size_t)line * L.P, S.piv, L, L.P);
  if (L.P <= 64) sep_x_line<2>(row, piv, L.P);
  else if (L.P <= 128) sep_x_line<4>(row, piv, L.P);
  else if (L.P <= 256) sep_x_line<8>(row, piv, L.P);
  else if (L.P <= 512) sep_x_line<16>(row, piv, L.P);
  else sep_x_line<32>(row, piv, L.P);
}

// -------------------------------------------------------------- kernels --
template <typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_init(Level<T> L, Sep<T> S, const T* __restrict__ b, T* __restrict__ x,
                                                       const PStore<T>* __restrict__ g, double* partials, SolveState* st,
                                                       cudaGraphConditionalHandle cond, int use_cond) {
  sep_init_body(L, S, b, x, g, partials, st, cond, use_cond, nullptr, vblock());
}
template <typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_update(Level<T> L, Sep<T> S, T* __restrict__ x, const T* d0, const T* d1,
                                                         const T* __restrict__ q, double* partials, SolveState* st,
                                                         cudaGraphConditionalHandle cond, int use_cond) {
  sep_update_body(L, S, x, d0, d1, q, partials, st, cond, use_cond, nullptr, vblock());
}
template <typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_zi(Level<T> L, Sep<T> S, T* __restrict__ z, double* partials,
                                                     SolveState* st) {
  sep_zi_body(L, S, z, partials, st, vblock());
}
template <bool INVERSE, typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_y(Level<T> L, Sep<T> S, const SolveState* st) {
  sep_y_body<INVERSE>(L, S, st, vblock());
}
template <typename T>
__global__ void __launch_bounds__(32 * SEP_X_LINES) k_sep_x(Level<T> L, Sep<T> S, const SolveState* st) {
  sep_x_body(L, S, st, vblock());
}

// ---------------------------------------------------------------- set-up --
// Eigenvector m of an axis of n cells at cell i.  Walls at both ends:
// cos(pi m (i + 1/2) / n).  An outlet at the high end: cos(theta (i + 1/2)),
// theta = (2m + 1) pi / (2n + 1), which vanishes at the ghost cell n; at the
// low end the same mirrored.
__device__ __forceinline__ double sep_mode(int m, int i, int n, bool out_lo, bool out_hi) {
  if (!out_lo && !out_hi) return sqrt((m == 0 ? 1.0 : 2.0) / n) * cospi((double)((long long)m * (2 * i + 1) % (4LL * n)) / (2.0 * n));
  if (out_lo) i = n - 1 - i;
  return 2.0 / sqrt(2.0 * n + 1.0) *
         cospi((double)((long long)(2 * m + 1) * (2 * i + 1) % (4LL * (2 * n + 1))) / (2.0 * (2 * n + 1)));
}
__device__ __forceinline__ double sep_eig(int m, int n, bool out_lo, bool out_hi) {
  const double s = (!out_lo && !out_hi) ? sinpi(m / (2.0 * n)) : sinpi((2 * m + 1) / (2.0 * (2 * n + 1)));
  return 4.0 * s * s;
}
// Matrices of an axis: forward (row mode, column cell) or transposed.  The
// halves of a folded axis: modes 0, 2, .. and 1, 3, .. at its first cells.
template <typename T>
__global__ void k_sep_pack(typename Sep<T>::Mat* A, SepAxis x, int out_lo, int out_hi, int transpose) {
  size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e >= sep_mat_count<T>(x)) return;
  A += e;
  const size_t ne = sep_block_count<T>(x.size(0));
  const int odd = e >= ne, m = x.size(odd);
  if (odd) e -= ne;
  auto val = [&](int r, int c) {
    if (r >= m || c >= m) return 0.0;
    const int mode = transpose ? c : r;
    return sep_mode(x.fold ? 2 * mode + odd : mode, transpose ? r : c, x.n, out_lo, out_hi);
  };
  if constexpr (sizeof(T) == 4) {
    const int KT = (m + 7) / 8, lane = (int)(e & 31), tile = (int)(e >> 5), g = lane >> 2, t = lane & 3;
    const int r0 = (tile / KT) * 16 + g, c0 = (tile % KT) * 8 + t;
    *A = make_float4((float)val(r0, c0), (float)val(r0 + 8, c0), (float)val(r0, c0 + 4), (float)val(r0 + 8, c0 + 4));
  } else {
    const int MP = (m + 1) & ~1;
    *A = val((int)(e % MP), (int)(e / MP));
  }
}
// Reciprocal pivots of the x systems, one line per thread, in FP64.
template <typename T>
__global__ void k_sep_pivots(Level<T> L, T* piv) {
  const int line = blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= L.ny * L.nz) return;
  const double lam = sep_eig(line % L.ny, L.ny, L.out_mask & 4, L.out_mask & 8) +
                     sep_eig(line / L.ny, L.nz, L.out_mask & 16, L.out_mask & 32);
  T* row = SEP_PTR(piv + (size_t)line * L.P, piv, L, L.P);
  double e = 0.0;
  for (int i = 0; i < L.nx; ++i) {
    double d = 2.0 + lam;
    if (i == 0 && !(L.out_mask & 1)) d -= 1.0;
    if (i == L.nx - 1 && !(L.out_mask & 2)) d -= 1.0;
    e = 1.0 / (d - e);
    row[i] = (T)e;
  }
}

}  // namespace uf
