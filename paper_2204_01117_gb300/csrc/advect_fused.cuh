// Fused MacCormack advection of the three velocity components (a2: Sec. 3,
// "Discretization and Numerical Integration", after Selle et al. 2008).
//
// One kernel runs both semi-Lagrangian passes.  A block owns a 32 x 8 column
// of lattice points (the same index range on the u, v and w lattices) and
// marches along z.  It stages, in shared memory:
//   * the time-level-n fields u, v, w on the column plus a halo of 2
//     (36 x 12 per plane, a ring of 8 planes per component, 5 of them live), copied one
//     plane ahead with cp.async;
//   * the forward-step values phi^ = phi(x - dt u(x)) of each component on
//     the column plus a halo of 1 (34 x 10 per plane, a ring of 4 planes, 3 live).
// The backward step, the correction phi* = phi^ + (phi - phi^(x + dt u(x)))/2
// and the clamp to the range of the forward sample's 8 values then read
// both from shared memory.  Per plane: two barriers (see advect_fused_body).
//
// The kernel is bound by the instructions it issues (shared-memory reads
// among them), so the common case is stripped to what it needs.  A thread
// forms phi^ of its own point of every component, keeping the displacements
// and ranges in registers for the backward step of the next plane, and of
// one fixed point of the halo (84 points x 3 components on 252 threads).
// While every displacement is below one cell the sample's cell follows from
// the signs of the displacements, its corners are staged, and only blocks and
// planes at the lattice's ends can clamp (EDGE).  The CFL time step keeps
// every displacement below cfl cells (FAR = false); a fixed time step need
// not, and a sample that leaves the cell then goes through the general
// functions below, each a call, which costs registers and moves even where
// it is never made: a kernel of its own (FAR = true).  Measured, FP32 and
// CFL time step, against general samples for all points, spread over the
// threads by component: 256 x 256 x 64 375 -> 164 us (310 M -> 139 M warp
// instructions, 1060 a cell), 512 x 512 x 128 2734 -> 1069 us; issue slots
// 77 % busy at 3 blocks per SM.
//
// Every value is formed by the same expressions as the two-kernel form
// (k_advect_forward, k_advect_backward) from the same inputs; only the
// memory the corners come from differs.  The results are bit for bit those
// of the two kernels.
//
// A sample whose corners are not all in the staged window reads global
// memory instead (a displacement of a cell or more, possible with a fixed
// time step); a backward sample whose corners are not all in the phi^ window
// recomputes phi^ at its corners from global memory.
//
// Tape (the adjoint's recompute sweep): when A.uh is not null, phi^ at every
// lattice point the block owns is also written to A.uh, A.vh, A.wh.
//
// When A.nut is not null the kernel also forms the eddy viscosity (a1) of
// the cells it owns from the staged time-level-n velocity, bit for bit what
// k_eddy_viscosity gives (strain_sq_acc rounds explicitly), which the step
// then does not launch.
#pragma once
#include "step_kernels.cuh"

namespace uf {

constexpr int MX = 32, MY = 8, MT = MX * MY;                    // owned column, threads per block
constexpr int MWX = MX + 4, MWY = MY + 4, MWP = MWX * MWY;      // window of the fields (halo 2)
constexpr int MHX = MX + 2, MHY = MY + 2, MHP = MHX * MHY;      // window of phi^ (halo 1)
constexpr int MHALO = MHP - MT;                                 // its points outside the column
static_assert(3 * MHALO <= MT, "one halo point per thread");
// ring depths (planes): 5 and 3 are live; powers of two make the slot of plane
// kk (kk >= -2) a bit mask instead of a division
constexpr int MFR = 8, MHR = 4;
constexpr int CF = MFR * MWP, CH = MHR * MHP;   // from one component's ring to the next
static_assert((MFR & (MFR - 1)) == 0 && (MHR & (MHR - 1)) == 0, "ring depths are powers of two");
#ifndef UF_ADVECT_MINB
#define UF_ADVECT_MINB 3   // resident blocks per SM the register budget is sized for
#endif

template <typename T>
constexpr size_t advect_fused_smem_total() {
  return sizeof(T) * 3 * ((size_t)MFR * MWP + (size_t)MHR * MHP);
}

// The block's shared memory: the rings of the fields ([3][MFR][MWP]), then
// those of phi^ ([3][MHR][MHP]).  A place in it is a byte offset into this
// one array: a 32-bit address that takes constant distances as immediates.
template <typename T>
__device__ __forceinline__ T* adv_sm(int place) {
  extern __shared__ __align__(16) unsigned char adv_smem[];
  return reinterpret_cast<T*>(adv_smem + place);
}

// Staged planes [zlo, zhi] of a W x H window with lattice origin (ox, oy),
// held in a ring of R planes (R a power of two: plane kk in slot kk & (R - 1)).
template <typename T, int W, int H, int R>
struct Win {
  int ring;   // place (bytes) of its first plane
  int ox, oy, zlo, zhi;
  __device__ __forceinline__ const T* plane(int kk) const { return adv_sm<T>(ring) + (kk & (R - 1)) * (W * H); }
  __device__ __forceinline__ bool holds(int i0, int i1, int j0, int j1, int k0, int k1) const {
    return i0 >= ox && i1 < ox + W && j0 >= oy && j1 < oy + H && k0 >= zlo && k1 <= zhi;
  }
  __device__ __forceinline__ void corners(int i0, int i1, int j0, int j1, int k0, int k1, T (&f)[8]) const {
    const T* p0 = plane(k0);
    const T* p1 = plane(k1);
    const int x0 = i0 - ox, x1 = i1 - ox, r0 = W * (j0 - oy), r1 = W * (j1 - oy);
    f[0] = p0[r0 + x0]; f[1] = p0[r0 + x1]; f[2] = p0[r1 + x0]; f[3] = p0[r1 + x1];
    f[4] = p1[r0 + x0]; f[5] = p1[r0 + x1]; f[6] = p1[r1 + x0]; f[7] = p1[r1 + x1];
  }
};

// Per-component accessors (Q known at compile time).
template <int Q, typename T>
__device__ __forceinline__ const Lattice& lat_of(const AdvectArgs<T>& A) { return Q == 0 ? A.Lu : (Q == 1 ? A.Lv : A.Lw); }
template <int Q, typename T>
__device__ __forceinline__ const T* field_of(const AdvectArgs<T>& A) { return Q == 0 ? A.u : (Q == 1 ? A.v : A.w); }
template <int Q, typename T>
__device__ __forceinline__ T* fhat_of(const AdvectArgs<T>& A) { return Q == 0 ? A.uh : (Q == 1 ? A.vh : A.wh); }
template <int Q, typename T>
__device__ __forceinline__ T* out_of(const AdvectArgs<T>& A) { return Q == 0 ? A.ut : (Q == 1 ? A.vt : A.wt); }

// Asynchronous copy of one value global -> shared (cp.async, L1-allocating).
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(sizeof(T)));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }

// A thread's two positions of the staged window (t, t + MT): offsets within
// a lattice plane (the u lattice; v, w and cells share theirs) and which
// lattices hold them (bits 0..2: u, v, w).
struct StagePos {
  int u[2], c[2], ok[2];
};
template <typename T>
__device__ __forceinline__ StagePos stage_pos(const AdvectArgs<T>& A, int i0, int j0) {
  StagePos S;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t = threadIdx.x + h * MT;
    const int gx = i0 - 2 + t % MWX, gy = j0 - 2 + t / MWX;
    const bool in = t < MWP && gx >= 0 && gy >= 0;
    S.u[h] = gx + A.Lu.P * gy;
    S.c[h] = gx + A.Lv.P * gy;
    S.ok[h] = !in ? 0 : (gx < A.Lu.Lx && gy < A.Lu.Ly ? 1 : 0) | (gx < A.Lv.Lx && gy < A.Lv.Ly ? 2 : 0) |
                            (gx < A.Lw.Lx && gy < A.Lw.Ly ? 4 : 0);
  }
  return S;
}
// Starts the copy of plane kk of the three fields into its ring slot.
template <typename T>
__device__ __forceinline__ void stage_plane(const AdvectArgs<T>& A, const StagePos& S, int kk) {
  if (kk < 0 || kk > A.nz) return;
  T* dst = adv_sm<T>(0) + (kk & (MFR - 1)) * MWP + threadIdx.x;
  const T* su = A.u + (size_t)kk * ((size_t)A.Lu.P * A.Lu.Ly);
  const T* sv = A.v + (size_t)kk * ((size_t)A.Lv.P * A.Lv.Ly);
  const T* sw = A.w + (size_t)kk * ((size_t)A.Lw.P * A.Lw.Ly);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (kk < A.nz) {
      if (S.ok[h] & 1) cp_async_elem(dst + h * MT, UF_PTR(su + S.u[h], A.u, A.Lu.P, A.Lu.Ly, A.Lu.Lz, 1, BA_U));
      if (S.ok[h] & 2) cp_async_elem(dst + MFR * MWP + h * MT, UF_PTR(sv + S.c[h], A.v, A.Lv.P, A.Lv.Ly, A.Lv.Lz, 1, BA_V));
    }
    if (S.ok[h] & 4) cp_async_elem(dst + 2 * MFR * MWP + h * MT, UF_PTR(sw + S.c[h], A.w, A.Lw.P, A.Lw.Ly, A.Lw.Lz, 1, BA_CW));
  }
}

// ------------------------------------------------- displacements < 1 cell --
// The cell of a sample at (index + off), |off| < 1, relative to the index: o
// = -1 below it, 0 above, and the weight t -- what axis_cell gives.  At the
// lattice's first (last) point a sample outside clamps to it.
template <bool EDGE, typename T>
__device__ __forceinline__ bool axis_near(T off, bool first, bool last, bool thin, T& t) {   // true: o = -1
  const bool below = off < T(0);
  t = below ? off + T(1) : off;
  if (!EDGE) return below;
  if (first && below) { t = T(0); return false; }
  if (last && !below) { t = thin ? T(0) : T(1); return !thin; }
  return below;
}
// Where a point lies on its lattice (EDGE only): the ends along each axis,
// and a lattice one point high.
struct Ends {
  bool x0, x1, y0, y1, z0, z1, thin;
};
__device__ __forceinline__ Ends ends_of(const Lattice& L, int gi, int gj, int k) {
  return Ends{gi == 0, gi == L.Lx - 1, gj == 0, gj == L.Ly - 1, k == 0, k == L.Lz - 1, L.Lz < 2};
}
// Trilinear sample around a staged point; pm, pc, pp: the point's place in
// the planes below, its own and above.
template <bool EDGE, bool RANGE, int W, typename T>
__device__ __forceinline__ T near_sample(int pm, int pc, int pp, T ox, T oy, T oz, const Ends& E, T* mn, T* mx) {
  T ta, tb, tc;
  const bool bx = axis_near<EDGE>(ox, E.x0, E.x1, false, ta);
  const bool by = axis_near<EDGE>(oy, E.y0, E.y1, false, tb);
  const bool bz = axis_near<EDGE>(oz, E.z0, E.z1, E.thin, tc);
  constexpr int B = sizeof(T);
  const int o = (bx ? -B : 0) + (by ? -W * B : 0);
  const T* q0 = adv_sm<T>((bz ? pm : pc) + o);
  const T* q1 = adv_sm<T>((bz || (EDGE && E.thin) ? pc : pp) + o);
  const T f[8] = {q0[0], q0[1], q0[W], q0[W + 1], q1[0], q1[1], q1[W], q1[W + 1]};
  return trilerp<T, RANGE>(f, ta, tb, tc, mn, mx);
}
template <typename T>
__device__ __forceinline__ bool below_one(const T (&d)[3]) {
  return max3(fabs(d[0]), fabs(d[1]), fabs(d[2])) < T(1);   // (a single NaN passes: its sample's corners are still the point's own)
}

// What a point's forward step leaves for its backward step: displacement and
// range of the forward sample's 8 values.
template <typename T>
struct Kept {
  T d[3], mn, mx;
};

// Forward sample with a displacement of a cell or more (or not a number):
// the general sample, from the staged window where it holds the corners.
// (By value: an address passed to a function that is not inlined would keep
// the range of every point in local memory.)
template <typename T>
struct Sampled {
  T val, mn, mx;
};
template <typename T>
__device__ __noinline__ Sampled<T> fwd_far(const T* __restrict__ F, Lattice L, Win<T, MWX, MWY, MFR> Wn, int i, int j, int k,
                                           T dx, T dy, T dz) {
  int i0, i1, j0, j1, k0, k1;
  T ta, tb, tc;
  axis_cell(i, -dx, L.Lx, i0, i1, ta);
  axis_cell(j, -dy, L.Ly, j0, j1, tb);
  axis_cell(k, -dz, L.Lz, k0, k1, tc);
  T f[8];
  if (Wn.holds(i0, i1, j0, j1, k0, k1)) Wn.corners(i0, i1, j0, j1, k0, k1, f);
  else corners_global(F, L, i0, i1, j0, j1, k0, k1, f);
  Sampled<T> r;
  r.val = trilerp<T, true>(f, ta, tb, tc, &r.mn, &r.mx);
  return r;
}
// phi^ at a lattice point from global memory only: the forward step of
// advect_forward_body.
template <typename T>
__device__ __noinline__ T fh_global(const AdvectArgs<T>& A, int q, Lattice L, const T* __restrict__ F, int i, int j,
                                    int k, T s) {
  T d[3];
  displacement(A, q, i, j, k, s, d);
  return sample<T, false>(F, L, i, -d[0], j, -d[1], k, -d[2]);
}
// Backward sample with a displacement of a cell or more: from the phi^
// window where it holds the corners, else phi^ is formed there again.
template <typename T>
__device__ __noinline__ T bwd_far(const AdvectArgs<T>& A, int q, Lattice L, const T* __restrict__ F,
                                  Win<T, MHX, MHY, MHR> Hw, int i, int j, int k, T dx, T dy, T dz, T s) {
  int a0, a1, b0, b1, c0, c1;
  T ta, tb, tc;
  axis_cell(i, dx, L.Lx, a0, a1, ta);
  axis_cell(j, dy, L.Ly, b0, b1, tb);
  axis_cell(k, dz, L.Lz, c0, c1, tc);
  T f[8];
  if (Hw.holds(a0, a1, b0, b1, c0, c1)) {
    Hw.corners(a0, a1, b0, b1, c0, c1, f);
  } else {
    for (int e = 0; e < 8; ++e) f[e] = fh_global(A, q, L, F, e & 1 ? a1 : a0, e & 2 ? b1 : b0, e & 4 ? c1 : c0, s);
  }
  return trilerp<T, false>(f, ta, tb, tc, nullptr, nullptr);
}

// A block's march: where it is and its shared memory.
template <typename T>
struct Advance {
  int i0, j0, k0, kend;
  T s;     // dt / h
  static constexpr int B = sizeof(T);
  // place of position b of plane kk in the window of component 0; the others lie CF (CH) values further on
  __device__ __forceinline__ int F(int kk, int b) const { return ((kk & (MFR - 1)) * MWP + b) * B; }
  __device__ __forceinline__ int H(int kk, int h) const { return (3 * CF + (kk & (MHR - 1)) * MHP + h) * B; }
};
// A point's place in three staged planes of the fields, and the pairs of
// faces around it: the sums of displacement(), each along its component's
// own axis.
template <typename T>
struct Near {
  int m, c, p;   // planes k - 1, k, k + 1
  __device__ __forceinline__ T at(int q, int e) const { return adv_sm<T>(q)[e]; }   // e values past place q
  __device__ __forceinline__ T u2(int q) const { return add_rn(at(q, 0), at(q, 1)); }
  __device__ __forceinline__ T v2(int q) const { return add_rn(at(q, CF), at(q, CF + MWX)); }
  __device__ __forceinline__ T w2(int o) const { return add_rn(at(c + o, 2 * CF), at(p + o, 2 * CF)); }
};
// Neighbour offsets of displacement(): the pair below and the pair above a
// face along x and y; along z the planes (EDGE: beyond the lattice's end the
// last pair).
template <bool EDGE, int B>
struct Around {   // in bytes
  int xl, xh, yl, yh;
  __device__ __forceinline__ Around(int gi, int gj, int nx, int ny)
      : xl(EDGE && gi == 0 ? 0 : -B), xh(EDGE && gi == nx ? -B : 0), yl(EDGE && gj == 0 ? 0 : -MWX * B),
        yh(EDGE && gj == ny ? -MWX * B : 0) {}
};

template <int Q, typename T>
__device__ __forceinline__ bool on_lattice(const AdvectArgs<T>& A, int gi, int gj, int m) {
  const Lattice& L = lat_of<Q>(A);
  return gi >= 0 && gj >= 0 && m >= 0 && gi < L.Lx && gj < L.Ly && m < L.Lz;
}

// phi^ at lattice point (gi, gj, m) of component q from its displacement.
template <bool EDGE, bool FAR, typename T>
__device__ __forceinline__ T forward_at(const AdvectArgs<T>& A, const Advance<T>& M, const Lattice& L, const T* F, int q, const Near<T>& N,
                                        int gi, int gj, int m, Kept<T>& K) {
  constexpr int B = sizeof(T);
  if (!FAR || below_one(K.d))
    return near_sample<EDGE, true, MWX>(N.m + q * CF * B, N.c + q * CF * B, N.p + q * CF * B, -K.d[0], -K.d[1], -K.d[2], ends_of(L, gi, gj, m), &K.mn,
                                        &K.mx);
  const Sampled<T> r = fwd_far(F, L, Win<T, MWX, MWY, MFR>{q * CF * B, M.i0 - 2, M.j0 - 2, max(m, M.k0) - 2, m + 1}, gi, gj, m,
                               K.d[0], K.d[1], K.d[2]);
  K.mn = r.mn;
  K.mx = r.mx;
  return r.val;
}
// Writes phi^ of an owned lattice point to the tape: inside the column, or
// the lattice's last point beyond it.
template <typename T>
__device__ __forceinline__ void tape_point(const AdvectArgs<T>& A, const Advance<T>& M, T* tape, const Lattice& L, int gi, int gj, int m, T val) {
  const bool ox = (gi >= M.i0 && gi < M.i0 + MX) || (gi >= M.i0 + MX && M.i0 + MX >= A.nx);
  const bool oy = (gj >= M.j0 && gj < M.j0 + MY) || (gj >= M.j0 + MY && M.j0 + MY >= A.ny);
  const bool oz = (m >= M.k0 && m < M.kend) || (m >= M.kend && M.kend == A.nz);
  UF_BOUNDS(!(ox && oy && oz) || (gi < L.Lx && gj < L.Ly && m < L.Lz), BA_LATTICE, gi, gj, m);
  if (ox && oy && oz) tape[(size_t)gi + (size_t)L.P * ((size_t)gj + (size_t)L.Ly * m)] = val;
}

// A thread's places: its own point and its halo point.
struct Places {
  int gi, gj, b, h;        // own point, its place in the two windows
  int hq, hi, hj, hb, hh;  // halo point: component (3: none), lattice point, places
};
__device__ __forceinline__ Places block_places(int i0, int j0) {
  Places X;
  const int t = threadIdx.x, tx = t % MX, ty = t / MX;
  X.gi = i0 + tx;
  X.gj = j0 + ty;
  X.b = (tx + 2) + MWX * (ty + 2);
  X.h = (tx + 1) + MHX * (ty + 1);
  X.hq = t / MHALO;
  const int e = t % MHALO;   // first row, last row, then the two side columns
  const int wx = e < MHX ? e : (e < 2 * MHX ? e - MHX : ((e & 1) ? MHX - 1 : 0));
  const int wy = e < MHX ? 0 : (e < 2 * MHX ? MHY - 1 : 1 + (e - 2 * MHX) / 2);
  X.hi = i0 - 1 + wx;
  X.hj = j0 - 1 + wy;
  X.hb = (wx + 1) + MWX * (wy + 1);
  X.hh = wx + MHX * wy;
  return X;
}

// phi^ on plane m: the thread's own point of every component (kept in K) and
// its halo point; stored (0 off the lattice), taped.  All loads come before
// the first store, so that the faces the components share are read once.
template <bool EDGE, bool FAR, typename T>
__device__ __forceinline__ void fhat_plane(const AdvectArgs<T>& A, const Advance<T>& M, const Places& X, int m, Kept<T> (&K)[3]) {
  const T s = M.s, s4 = T(0.25) * s;
  const int za = EDGE ? max(m - 1, 0) : m - 1, zc = EDGE ? min(m, A.nz - 1) : m;   // cell planes below and above the w point
  {
    const Near<T> N{M.F(m - 1, X.b), M.F(m, X.b), M.F(m + 1, X.b)};
    const Around<EDGE, sizeof(T)> o(X.gi, X.gj, A.nx, A.ny);
    const int a = EDGE ? M.F(za, X.b) : N.m, c = EDGE ? M.F(zc, X.b) : N.c;
    const bool on0 = !EDGE || on_lattice<0>(A, X.gi, X.gj, m), on1 = !EDGE || on_lattice<1>(A, X.gi, X.gj, m),
               on2 = !EDGE || on_lattice<2>(A, X.gi, X.gj, m);
    T val[3] = {T(0), T(0), T(0)};
    if (on0) {
      K[0].d[0] = s * N.at(N.c, 0);
      K[0].d[1] = s4 * add_rn(N.v2(N.c + o.xl), N.v2(N.c + o.xh));
      K[0].d[2] = s4 * add_rn(N.w2(o.xl), N.w2(o.xh));
      val[0] = forward_at<EDGE, FAR>(A, M, A.Lu, A.u, 0, N, X.gi, X.gj, m, K[0]);
    }
    if (on1) {
      K[1].d[0] = s4 * add_rn(N.u2(N.c + o.yl), N.u2(N.c + o.yh));
      K[1].d[1] = s * N.at(N.c, CF);
      K[1].d[2] = s4 * add_rn(N.w2(o.yl), N.w2(o.yh));
      val[1] = forward_at<EDGE, FAR>(A, M, A.Lv, A.v, 1, N, X.gi, X.gj, m, K[1]);
    }
    if (on2) {
      K[2].d[0] = s4 * add_rn(N.u2(a), N.u2(c));
      K[2].d[1] = s4 * add_rn(N.v2(a), N.v2(c));
      K[2].d[2] = s * N.at(N.c, 2 * CF);
      val[2] = forward_at<EDGE, FAR>(A, M, A.Lw, A.w, 2, N, X.gi, X.gj, m, K[2]);
    }
    T* h = adv_sm<T>(M.H(m, X.h));
    h[0] = val[0];
    h[CH] = val[1];
    h[2 * CH] = val[2];
    if (A.uh) {
      if (on0 && m >= 0) tape_point(A, M, A.uh, A.Lu, X.gi, X.gj, m, val[0]);
      if (on1 && m >= 0) tape_point(A, M, A.vh, A.Lv, X.gi, X.gj, m, val[1]);
      if (on2 && m >= 0) tape_point(A, M, A.wh, A.Lw, X.gi, X.gj, m, val[2]);
    }
  }
  if (X.hq < 3) {
    const Near<T> N{M.F(m - 1, X.hb), M.F(m, X.hb), M.F(m + 1, X.hb)};
    const Around<EDGE, sizeof(T)> o(X.hi, X.hj, A.nx, A.ny);
    const Lattice& L = X.hq == 0 ? A.Lu : (X.hq == 1 ? A.Lv : A.Lw);
    T val = T(0);
    if (!EDGE || (X.hi >= 0 && X.hj >= 0 && m >= 0 && X.hi < L.Lx && X.hj < L.Ly && m < L.Lz)) {
      Kept<T> K1;
      const T own = s * N.at(N.c, X.hq * CF);
      if (X.hq == 0) {
        K1.d[0] = own;
        K1.d[1] = s4 * add_rn(N.v2(N.c + o.xl), N.v2(N.c + o.xh));
        K1.d[2] = s4 * add_rn(N.w2(o.xl), N.w2(o.xh));
      } else if (X.hq == 1) {
        K1.d[0] = s4 * add_rn(N.u2(N.c + o.yl), N.u2(N.c + o.yh));
        K1.d[1] = own;
        K1.d[2] = s4 * add_rn(N.w2(o.yl), N.w2(o.yh));
      } else {
        const int a = EDGE ? M.F(za, X.hb) : N.m, c = EDGE ? M.F(zc, X.hb) : N.c;
        K1.d[0] = s4 * add_rn(N.u2(a), N.u2(c));
        K1.d[1] = s4 * add_rn(N.v2(a), N.v2(c));
        K1.d[2] = own;
      }
      const T* F = X.hq == 0 ? A.u : (X.hq == 1 ? A.v : A.w);
      val = forward_at<EDGE, FAR>(A, M, L, F, X.hq, N, X.hi, X.hj, m, K1);
      if (A.uh) tape_point(A, M, X.hq == 0 ? A.uh : (X.hq == 1 ? A.vh : A.wh), L, X.hi, X.hj, m, val);
    }
    adv_sm<T>(M.H(m, X.hh))[X.hq * CH] = val;
  }
}

// Backward step, correction and clamp of component Q at the thread's own
// point on plane k: phi* = phi^ + (phi - phi^(x + dt u(x)))/2, clamped.  f:
// the point in the staged plane k; hm, hc, hp: in the phi^ planes around it.
template <int Q, bool EDGE, bool FAR, typename T>
__device__ __forceinline__ void maccormack_point(const AdvectArgs<T>& A, const Advance<T>& M, const Places& X, int k, int f, int hm,
                                                 int hc, int hp, const Kept<T>& K) {
  const int gi = X.gi, gj = X.gj;
  if (EDGE) {
    const bool interior = Q == 0 ? (gi > 0 && gi < A.nx && gj < A.ny)
                                 : (Q == 1 ? (gi < A.nx && gj > 0 && gj < A.ny) : (gi < A.nx && gj < A.ny && k > 0 && k < A.nz));
    if (!interior) return;
  }
  const Lattice& L = lat_of<Q>(A);
  constexpr int B = sizeof(T);
  T bwd;
  if (!FAR || below_one(K.d))
    bwd = near_sample<EDGE, false, MHX>(hm + Q * CH * B, hc + Q * CH * B, hp + Q * CH * B, K.d[0], K.d[1], K.d[2], ends_of(L, gi, gj, k),
                                        (T*)nullptr, (T*)nullptr);
  else
    bwd = bwd_far(A, Q, L, field_of<Q>(A), Win<T, MHX, MHY, MHR>{(3 * CF + Q * CH) * B, M.i0 - 1, M.j0 - 1, k - 1, k + 1}, gi, gj, k, K.d[0],
                  K.d[1], K.d[2], M.s);
  const T fwd = adv_sm<T>(hc)[Q * CH], own = adv_sm<T>(f)[Q * CF];
  const T r = fwd + T(0.5) * (own - bwd);
  *UF_PTR(out_of<Q>(A) + (size_t)k * ((size_t)L.P * L.Ly) + (gi + L.P * gj), out_of<Q>(A), L.P, L.Ly, L.Lz, 1, BA_LATTICE) =
      fmin(fmax(r, K.mn), K.mx);
}
template <bool EDGE, bool FAR, typename T>
__device__ __forceinline__ void maccormack_plane(const AdvectArgs<T>& A, const Advance<T>& M, const Places& X, int k,
                                                 const Kept<T> (&K)[3]) {
  const int f = M.F(k, X.b), hm = M.H(k - 1, X.h), hc = M.H(k, X.h), hp = M.H(k + 1, X.h);
  maccormack_point<0, EDGE, FAR>(A, M, X, k, f, hm, hc, hp, K[0]);
  maccormack_point<1, EDGE, FAR>(A, M, X, k, f, hm, hc, hp, K[1]);
  maccormack_point<2, EDGE, FAR>(A, M, X, k, f, hm, hc, hp, K[2]);
}

// Eddy viscosity of the thread's cell on plane k (the expressions of
// eddy_viscosity_body) with the faces strain_sq reads taken from the staged
// windows: planes k-1 .. k+2 of the fields are complete here.
template <bool EDGE, typename T>
__device__ __forceinline__ void eddy_point(const AdvectArgs<T>& A, const Advance<T>& M, const Places& X, int k, const T* kf,
                                           const T* om, T cap) {
  const int fm = M.F(k - 1, X.b), fc = M.F(k, X.b), fp = M.F(k + 1, X.b);
  const T S2 = strain_sq_acc<EDGE, T>(
      A.sp, X.gi, X.gj, k, [&](int q, int dx, int dy, int dz) { return adv_sm<T>(dz == 0 ? fc : (dz < 0 ? fm : fp))[q * CF + dx + MWX * dy]; });
  const size_t plane = (size_t)k * ((size_t)A.Lw.P * A.Lw.Ly);   // (cells share the w lattice's rows)
  const int c = X.gi + A.Lw.P * X.gj;
  auto cell = [&](auto* f) { return UF_PTR(f + plane + c, f, A.Lw.P, A.Lw.Ly, A.nz, 1, BA_CW); };
  *cell(A.nut) = limited_nut(A.sp, *cell(kf), *cell(om), S2, cap);
}

// Pipeline per plane m of phi^:  wait for plane m+1 of the fields, sync,
// start the copy of plane m+2 (into the slot of m-6, which no one reads any
// more), phi^ of plane m, sync, phi* of plane m-1.  The phi^ phase reads
// the fields on planes [m-2, m+1].  kf, om: k and omega of the eddy
// viscosity (where A.nut is set).
template <bool FAR, typename T>
__device__ __forceinline__ void advect_fused_body(const AdvectArgs<T>& A, int zc, const T* kf, const T* om, const VBlock& vb) {
  Advance<T> M;
  M.i0 = vb.x * MX;
  M.j0 = vb.y * MY;
  M.k0 = vb.z * zc;
  M.kend = min(A.nz, M.k0 + zc);
  M.s = *A.dtT * A.inv_h;
  const StagePos S = stage_pos(A, M.i0, M.j0);
  for (int kk = M.k0 - 2; kk <= M.k0; ++kk) stage_plane(A, S, kk);
  cp_async_commit();
  const Places X = block_places(M.i0, M.j0);
  // every point of the phi^ window, its samples and its faces inside all three lattices along x and y
  const bool inner = M.i0 >= 2 && M.i0 + MX <= A.nx - 2 && M.j0 >= 2 && M.j0 + MY <= A.ny - 2;
  auto edge = [&](int m) { return !inner || m < 1 || m > A.nz - 2; };
  const T cap = A.nut ? nut_cap(A.sp, *A.dtT) : T(0);
  Kept<T> K[3], N[3];
  // m: the plane of phi^; phi* follows one plane behind.  (One copy of each
  // phase's code in the loop: the kernel is sensitive to its code size.)
  for (int m = M.k0 - 1; m <= M.kend; ++m) {
    const int k = m - 1;
    cp_async_wait_all();
    __syncthreads();
    stage_plane(A, S, m + 2);
    cp_async_commit();
    if (edge(m)) fhat_plane<true, FAR>(A, M, X, m, N);
    else fhat_plane<false, FAR>(A, M, X, m, N);
    if (m > M.k0) {
      __syncthreads();
      if (edge(k)) maccormack_plane<true, FAR>(A, M, X, k, K);
      else maccormack_plane<false, FAR>(A, M, X, k, K);
      if (A.nut && X.gi < A.nx && X.gj < A.ny) {
        if (edge(k)) eddy_point<true>(A, M, X, k, kf, om, cap);
        else eddy_point<false>(A, M, X, k, kf, om, cap);
      }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) K[q] = N[q];
  }
  cp_async_wait_all();
}

template <typename T, bool FAR>
__global__ void __launch_bounds__(MT, FAR ? 2 : UF_ADVECT_MINB) k_advect_fused(const __grid_constant__ AdvectArgs<T> A, int zc) {
  advect_fused_body<FAR, T>(A, zc, A.kf, A.om, vblock());
}

}  // namespace uf
