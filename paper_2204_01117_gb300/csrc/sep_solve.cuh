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
// (k_sep_zf, k_sep_y, k_sep_x, k_sep_y, k_sep_zi).  (Lynch, Rice and Thomas,
// "Direct solution of partial difference equations by tensor product
// methods", Numer. Math. 6, 1964.)
//
// In FP32 the inverse is exact to rounding, which leaves CG one or two
// iterations to 1e-7 where the V-cycle needs seven to eleven, and an
// application is 5 launches where the V-cycle has 14 to 18 that depend on
// one another.  CG still stops on ||r|| <= tol ||b|| with FP64 inner products,
// so the solution is the same to the same tolerance; its error against 64
// bits is at most the V-cycle's (512 x 512 x 128, w after two steps: 2.2e-6
// against 4.8e-6).  Measured on a GB300, one time step with the V-cycle and
// with this: 48 x 40 x 16 0.73 -> 0.20 ms, 157 x 203 x 41 1.87 -> 0.47 ms,
// 256 x 256 x 64 2.20 -> 1.09 ms, 512 x 768 x 1 1.24 -> 0.34 ms,
// 512 x 512 x 128 13.0 -> 8.7 ms (where the y transforms, 2 n^2 per column
// and pass, take 0.41 ms each); the longest axes that fit were all faster.
//
// The transforms are contractions of a field with a constant n x n matrix:
// tensor cores, TF32 operands split into a high and a low part (x = hi + lo,
// 11 bits each), three products hi hi + hi lo + lo hi accumulated in FP32.
// The dropped lo lo is below 2^-22 of the product, so a transform is about
// as accurate as one in plain FP32.
#pragma once
#include "mg_fused.cuh"

namespace uf {

constexpr int SEP_T = 256;        // threads of the transform kernels (8 warps)
constexpr int SEP_X_LINES = 8;    // lines (warps) per block of the x solve
constexpr int SEP_MAX_NX = 1024;  // 32 lanes x 32 values per line

// FP64 grids do the same on the FP64 pipe, 1/64 of the FP32 rate on this
// chip: the products are then what a pass costs, and a rule on the sizes
// keeps the V-cycle where they would outweigh the iterations saved
// (sep_available in capi.cu, with both sides measured).
template <typename T>
struct SepMat { using type = float4; };   // FP32: see below
template <>
struct SepMat<double> { using type = double; };

// Separable solver of one grid.  FP32 matrices are packed in the order in
// which the lanes of a warp read the A operand of mma.m16n8k8: one float4 per
// lane and 16 x 8 tile, tiles row by row, zero beyond the matrix.  FP64
// matrices are stored column by column, each padded with zeros to an even
// number of rows.
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
// Columns of a y panel in units of 32: two while it fits (n <= 768), else one.
constexpr int SEP_Y_WIDE = 768;
template <typename T>
__host__ __device__ inline int sep_y_wn(int ny) { return sizeof(T) == 4 && ny <= SEP_Y_WIDE ? 2 : 1; }
template <typename T>
constexpr int SEP_Z_WN = sizeof(T) == 4 ? 4 : 1;
template <typename T>
inline size_t sep_smem(int wn, int n) { return sizeof(T) * (size_t)((n + 7) / 8 * 8) * (sizeof(T) == 4 ? 32 * wn + 8 : 32); }
// Columns (x, y) of a z panel, and the blocks that cover the plane.  One cell
// in z has nothing to transform: the threads just share the columns out.
template <typename T>
__host__ __device__ inline int sep_z_cols(int nz) { return nz > 1 ? 32 * SEP_Z_WN<T> : (int)(16 / sizeof(T)) * SEP_T; }
template <typename T>
inline unsigned sep_z_blocks(int P, int ny, int nz) {
  return (unsigned)(((size_t)P * ny + sep_z_cols<T>(nz) - 1) / sep_z_cols<T>(nz));
}
// Blocks that share a y panel, each taking every split-th round of result
// rows: a quasi-2D grid has fewer panels than SMs (512 x 768 x 1: 8, one pass
// 97 us unsplit, 27 us split).
constexpr int SEP_Y_BLOCKS = 304;   // two resident blocks on each of 152 SMs
template <typename T>
__host__ __device__ inline int sep_y_split(int P, int ny, int nz) {
  const int wn = sep_y_wn<T>(ny), rows = sizeof(T) == 4 ? 32 * (8 / wn) : 32;   // of a round
  const int panels = (P + 32 * wn - 1) / (32 * wn) * nz, rounds = (ny + rows - 1) / rows;
  const int want = (SEP_Y_BLOCKS + panels - 1) / panels;
  return want < rounds ? want : rounds;
}
// 16 bytes of a field.
template <typename T>
struct alignas(16) SepVec {
  static constexpr int N = 16 / sizeof(T);
  T e[N];
};

// x = hi + lo (+ below 2^-22 |x|): hi rounded to TF32's 11 bits, lo cut to them.
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

// Result rows of the block's panel: A (M x K packed) times sB ([K][pitch]),
// rounds part, part + parts, ... of 32 WM rows.
// put(row, column of the panel (even), value, next value).
template <int WN, typename Put>
__device__ __forceinline__ void sep_gemm(const float4* __restrict__ A, int M, int K, const float* sB, int part, int parts,
                                         Put put) {
  constexpr int PB = SEP_PITCH<float, WN>, WM = 8 / WN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3, wm = warp / WN, wn = warp % WN;
  const int KT = (K + 7) / 8, MT16 = (M + 15) / 16;
  const float* b = sB + t * PB + wn * 32 + g;
  for (int m0 = 2 * (wm + WM * part); m0 < MT16; m0 += 2 * WM * parts) {
    const bool two = m0 + 1 < MT16;
    const float4* a0 = A + (size_t)m0 * KT * 32 + lane;
    const float4* a1 = a0 + (two ? (size_t)KT * 32 : 0);
    float acc[2][4][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[h][n][e] = 0.f;
    float4 n0 = __ldg(a0), n1 = __ldg(a1);
#pragma unroll 2
    for (int kt = 0; kt < KT; ++kt) {
      const float4 c0 = n0, c1 = n1;
      if (kt + 1 < KT) {
        n0 = __ldg(a0 + (size_t)(kt + 1) * 32);
        n1 = __ldg(a1 + (size_t)(kt + 1) * 32);
      }
      uint32_t h0[4], l0[4], h1[4], l1[4];
      tf32_split(c0.x, h0[0], l0[0]); tf32_split(c0.y, h0[1], l0[1]);
      tf32_split(c0.z, h0[2], l0[2]); tf32_split(c0.w, h0[3], l0[3]);
      tf32_split(c1.x, h1[0], l1[0]); tf32_split(c1.y, h1[1], l1[1]);
      tf32_split(c1.z, h1[2], l1[2]); tf32_split(c1.w, h1[3], l1[3]);
      const float* bk = b + kt * 8 * PB;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        uint32_t bh0, bl0, bh1, bl1;
        tf32_split(bk[n * 8], bh0, bl0);
        tf32_split(bk[n * 8 + 4 * PB], bh1, bl1);
        mma_tf32(acc[0][n], l0, bh0, bh1);
        mma_tf32(acc[1][n], l1, bh0, bh1);
        mma_tf32(acc[0][n], h0, bl0, bl1);
        mma_tf32(acc[1][n], h1, bl0, bl1);
        mma_tf32(acc[0][n], h0, bh0, bh1);
        mma_tf32(acc[1][n], h1, bh0, bh1);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = (m0 + h) * 16 + g;
      if (h == 1 && !two) break;
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int col = wn * 32 + n * 8 + 2 * t;
        if (row < M) put(row, col, acc[h][n][0], acc[h][n][1]);
        if (row + 8 < M) put(row + 8, col, acc[h][n][2], acc[h][n][3]);
      }
    }
  }
}

// FP64: lane l owns columns 2 (l % 16), + 1 and rows 2 (l / 16), + 1 of its
// warp's four (A: column by column, MP rows each).
template <int WN, typename Put>
__device__ __forceinline__ void sep_gemm(const double* __restrict__ A, int M, int K, const double* sB, int part, int parts,
                                         Put put) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = 2 * (lane & 15), MP = (M + 1) & ~1;
  for (int r0 = 4 * warp + 32 * part; r0 < M; r0 += 32 * parts) {
    const int row = r0 + 2 * (lane >> 4);
    const double* a = A + (row < M ? row : 0);
    double c00 = 0, c01 = 0, c10 = 0, c11 = 0;
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const double2 av = __ldg(reinterpret_cast<const double2*>(a + (size_t)k * MP));
      const double2 bv = *reinterpret_cast<const double2*>(sB + k * 32 + col);
      c00 = fma(av.x, bv.x, c00);
      c01 = fma(av.x, bv.y, c01);
      c10 = fma(av.y, bv.x, c10);
      c11 = fma(av.y, bv.y, c11);
    }
    if (row < M) put(row, col, c00, c01);
    if (row + 1 < M) put(row + 1, col, c10, c11);
  }
}

__device__ __forceinline__ void sep_put2(float* o, float a, float b) { *reinterpret_cast<float2*>(o) = make_float2(a, b); }
__device__ __forceinline__ void sep_put2(double* o, double a, double b) { *reinterpret_cast<double2*>(o) = make_double2(a, b); }
__device__ __forceinline__ float2 sep_get2(const float* o) { return *reinterpret_cast<const float2*>(o); }
__device__ __forceinline__ double2 sep_get2(const double* o) { return *reinterpret_cast<const double2*>(o); }

// ------------------------------------------------------- z transforms ----
// A panel is 128 consecutive columns (x, y) of the P x ny plane with every z
// in shared memory, so each cell is read once.  CG = true (inside the CG
// loop): the panel's load is also the CG update x += alpha d, r -= alpha q
// with ||r||^2 and the convergence test.  Columns in the row padding
// (x >= nx) are forced to zero.
template <bool CG, typename T>
__device__ __forceinline__ void sep_zf_body(const Level<T>& L, const Sep<T>& S, T* __restrict__ x, const T* d0, const T* d1,
                                            const T* __restrict__ q, double* partials, SolveState* st,
                                            cudaGraphConditionalHandle cond, int use_cond, int* left, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  __shared__ double sh[32];
  __shared__ bool last;
  if (st->converged) return;
  using V = SepVec<T>;
  constexpr int WN = SEP_Z_WN<T>, BN = 32 * WN, PB = SEP_PITCH<T, WN>, VR = BN / V::N;
  static_assert(SEP_T % VR == 0, "a thread keeps its columns");
  const size_t PS = (size_t)L.P * L.ny;
  const bool flat = L.nz == 1;   // one cell in z: the identity, a thread per 16 bytes
  const int row0 = flat ? 0 : threadIdx.x / VR, col0 = V::N * (flat ? threadIdx.x : threadIdx.x % VR);
  const size_t c = (size_t)vb.x * sep_z_cols<T>(L.nz) + col0;
  const bool in = c < PS;
  const int left_x = L.nx - (int)(c % L.P);   // how many of the values lie inside the domain
  const int it0 = st->iter;
  const T alpha = CG ? (T)st->alpha : T(0);
  const T* dn = (it0 & 1) ? d0 : d1;
  DotAcc<T> dacc;
  const int KP = flat ? 1 : (L.nz + 7) / 8 * 8;
#pragma unroll 2
  for (int k = row0; k < KP; k += SEP_T / VR) {
    V v = {};
    if (in && k < L.nz) {
      const size_t o = (size_t)k * PS + c;
      v = *reinterpret_cast<const V*>(L.r + o);
      if (CG) {
        const V qv = *reinterpret_cast<const V*>(q + o);
        const V dv = *reinterpret_cast<const V*>(dn + o);
        V xv = *reinterpret_cast<const V*>(x + o);
#pragma unroll
        for (int e = 0; e < V::N; ++e) {
          v.e[e] = e < left_x ? v.e[e] - alpha * qv.e[e] : T(0);
          xv.e[e] = e < left_x ? xv.e[e] + alpha * dv.e[e] : T(0);
          dacc.add(v.e[e], v.e[e]);
        }
        *reinterpret_cast<V*>(L.r + o) = v;
        *reinterpret_cast<V*>(x + o) = xv;
      }
    }
    if (!flat) *reinterpret_cast<V*>(sep_sm + k * PB + col0) = v;
    else if (in) *reinterpret_cast<V*>(S.t + c) = v;
  }
  if (!flat) {
    __syncthreads();
    const size_t cb = (size_t)vb.x * BN;
    sep_gemm<WN>(S.zf, L.nz, L.nz, sep_sm, 0, 1, [&](int row, int col, T a, T b) {
      if (cb + col < PS) sep_put2(S.t + (size_t)row * PS + cb + col, a, b);
    });
  }
  if (CG) {
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
}

// Back along z: z = Qz^T t, and r.z (CG beta in mode 1).
template <typename T>
__device__ __forceinline__ void sep_zi_body(const Level<T>& L, const Sep<T>& S, T* __restrict__ z, int mode, double* partials,
                                            SolveState* st, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  __shared__ double sh[32];
  __shared__ bool last;
  if (st->converged) return;
  using V = SepVec<T>;
  constexpr int WN = SEP_Z_WN<T>, BN = 32 * WN, PB = SEP_PITCH<T, WN>, VR = BN / V::N;
  const size_t PS = (size_t)L.P * L.ny;
  const bool flat = L.nz == 1;
  const int col0 = V::N * (flat ? threadIdx.x : threadIdx.x % VR);
  const size_t c = (size_t)vb.x * sep_z_cols<T>(L.nz) + col0;
  DotAcc<T> dacc;
  auto put = [&](size_t o, T a, T b) {
    const auto rv = sep_get2(L.r + o);
    sep_put2(z + o, a, b);
    dacc.add(rv.x, a);
    dacc.add(rv.y, b);
  };
  if (flat) {
    if (c < PS) {
      const V v = *reinterpret_cast<const V*>(S.t + c);
#pragma unroll
      for (int e = 0; e < V::N; e += 2) put(c + e, v.e[e], v.e[e + 1]);
    }
  } else {
    const int KP = (L.nz + 7) / 8 * 8;
#pragma unroll 4
    for (int k = threadIdx.x / VR; k < KP; k += SEP_T / VR) {
      V v = {};
      if (c < PS && k < L.nz) v = *reinterpret_cast<const V*>(S.t + (size_t)k * PS + c);
      *reinterpret_cast<V*>(sep_sm + k * PB + col0) = v;
    }
    __syncthreads();
    const size_t cb = (size_t)vb.x * BN;
    sep_gemm<WN>(S.zi, L.nz, L.nz, sep_sm, 0, 1, [&](int row, int col, T a, T b) {
      if (cb + col < PS) put((size_t)row * PS + cb + col, a, b);
    });
  }
  const double vals[1] = {block_sum<SEP_T>(dacc.value(), sh)};
  if (publish_partials<1>(partials, &st->ticket[0], vals, &last, vb)) {
    double tot[1];
    reduce_partials_sum<SEP_T, 1>(partials, tot, sh, vb.n);
    if (threadIdx.x == 0) {
      finish_rz(st, tot[0], mode);
      st->ticket[0] = 0u;
    }
  }
}

// --------------------------------------------------------- y transforms --
// One panel of 32 WN columns of a z plane, every y; blocks vb.y of `split`
// share the panel's result rows.
template <int WN, typename T>
__device__ __forceinline__ void sep_y_panel(const Level<T>& L, const typename Sep<T>::Mat* A, const T* __restrict__ src,
                                            T* __restrict__ dst, int split, const VBlock& vb) {
  extern __shared__ __align__(16) unsigned char sep_raw[];
  T* sep_sm = reinterpret_cast<T*>(sep_raw);
  using V = SepVec<T>;
  constexpr int BN = 32 * WN, PB = SEP_PITCH<T, WN>, VR = BN / V::N;
  const int x0 = vb.x * BN, xv = V::N * (threadIdx.x % VR);
  const size_t base = (size_t)vb.z * L.P * L.ny + x0;
  const bool in = x0 + xv < L.P;
  const int KP = (L.ny + 7) / 8 * 8;
#pragma unroll 4
  for (int j = threadIdx.x / VR; j < KP; j += SEP_T / VR) {
    V v = {};
    if (in && j < L.ny) v = *reinterpret_cast<const V*>(src + base + (size_t)j * L.P + xv);
    *reinterpret_cast<V*>(sep_sm + j * PB + xv) = v;
  }
  __syncthreads();
  sep_gemm<WN>(A, L.ny, L.ny, sep_sm, vb.y, split, [&](int row, int col, T a, T b) {
    if (x0 + col < L.P) sep_put2(dst + base + (size_t)row * L.P + col, a, b);
  });
}
template <typename T>
__device__ __forceinline__ void sep_y_body(const Level<T>& L, const Sep<T>& S, int inverse, const SolveState* st,
                                           const VBlock& vb) {
  if (st->converged) return;
  const auto* A = inverse ? S.yi : S.yf;
  const T* src = inverse ? S.u : S.t;
  T* dst = inverse ? S.t : S.u;
  const int split = sep_y_split<T>(L.P, L.ny, L.nz);
  if (sizeof(T) == 4 && L.ny <= SEP_Y_WIDE) sep_y_panel<sizeof(T) == 4 ? 2 : 1>(L, A, src, dst, split, vb);
  else sep_y_panel<1>(L, A, src, dst, split, vb);
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
  using V = SepVec<T>;
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
  T* row = S.u + (size_t)line * L.P;
  const T* piv = S.piv + (size_t)line * L.P;
  if (L.P <= 64) sep_x_line<2>(row, piv, L.P);
  else if (L.P <= 128) sep_x_line<4>(row, piv, L.P);
  else if (L.P <= 256) sep_x_line<8>(row, piv, L.P);
  else if (L.P <= 512) sep_x_line<16>(row, piv, L.P);
  else sep_x_line<32>(row, piv, L.P);
}

// -------------------------------------------------------------- kernels --
template <bool CG, typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_zf(Level<T> L, Sep<T> S, T* __restrict__ x, const T* d0, const T* d1,
                                                     const T* __restrict__ q, double* partials, SolveState* st,
                                                     cudaGraphConditionalHandle cond, int use_cond) {
  sep_zf_body<CG>(L, S, x, d0, d1, q, partials, st, cond, use_cond, nullptr, vblock());
}
template <typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_zi(Level<T> L, Sep<T> S, T* __restrict__ z, int mode, double* partials,
                                                     SolveState* st) {
  sep_zi_body(L, S, z, mode, partials, st, vblock());
}
template <typename T>
__global__ void __launch_bounds__(SEP_T, 2) k_sep_y(Level<T> L, Sep<T> S, int inverse, const SolveState* st) {
  sep_y_body(L, S, inverse, st, vblock());
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
// Matrix of an axis: forward (row mode, column cell) or its transpose.
__device__ __forceinline__ double sep_entry(int r, int c, int n, int out_lo, int out_hi, int transpose) {
  if (r >= n || c >= n) return 0.0;
  return transpose ? sep_mode(c, r, n, out_lo, out_hi) : sep_mode(r, c, n, out_lo, out_hi);
}
template <typename T>
__host__ __device__ inline size_t sep_mat_count(int n) {   // elements of Sep<T>::Mat
  return sizeof(T) == 4 ? (size_t)((n + 15) / 16) * ((n + 7) / 8) * 32 : (size_t)n * ((n + 1) & ~1);
}
template <typename T>
__global__ void k_sep_pack(typename Sep<T>::Mat* A, int n, int out_lo, int out_hi, int transpose) {
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e >= sep_mat_count<T>(n)) return;
  if constexpr (sizeof(T) == 4) {
    const int KT = (n + 7) / 8, lane = (int)(e & 31), tile = (int)(e >> 5), g = lane >> 2, t = lane & 3;
    const int r0 = (tile / KT) * 16 + g, c0 = (tile % KT) * 8 + t;
    auto val = [&](int r, int c) { return (float)sep_entry(r, c, n, out_lo, out_hi, transpose); };
    A[e] = make_float4(val(r0, c0), val(r0 + 8, c0), val(r0, c0 + 4), val(r0 + 8, c0 + 4));
  } else {
    const int NP = (n + 1) & ~1;
    A[e] = sep_entry((int)(e % NP), (int)(e / NP), n, out_lo, out_hi, transpose);
  }
}
// Reciprocal pivots of the x systems, one line per thread, in FP64.
template <typename T>
__global__ void k_sep_pivots(Level<T> L, T* piv) {
  const int line = blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= L.ny * L.nz) return;
  const double lam = sep_eig(line % L.ny, L.ny, L.out_mask & 4, L.out_mask & 8) +
                     sep_eig(line / L.ny, L.nz, L.out_mask & 16, L.out_mask & 32);
  T* row = piv + (size_t)line * L.P;
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
