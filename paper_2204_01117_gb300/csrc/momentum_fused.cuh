// Fused diffusion, porosity drag, velocity BCs and pressure right-hand side
// (a3-a6: Eq. momen_drag's (nu + nu_t) lap u; the forward-Euler drag step
// and the BC rules of Sec. 3; b = -(rho h / dt) h div u).
//
// One z-marching kernel per 32 x 8 column of cells replaces k_diffuse,
// k_drag_bc and k_pressure_rhs.  Per block, in shared memory:
//   * the advected velocity (u~, v~, w~), nu_t and the drag coefficient c on
//     the column plus a halo of 2 (36 x 12, a ring of 4 planes), copied one
//     plane ahead with cp.async;
//   * the diffused velocity u2 of the three components on the column plus a
//     halo of 1 (34 x 10, a ring of 2 planes);
//   * the dragged velocity u3 of the plane's x and y faces, for the fluxes.
// Per plane k: u2 on plane k+1 and b of plane k-1 with ||b||^2, sync, u3 on
// the faces of plane k (u, v) and on the w faces of plane k+1, sync.
//
// Bound by the instructions it issues, as the advection, and built like it:
// a thread forms u2 of its own three faces, with their values on the planes
// below and at its own in registers, and of one fixed halo face; only blocks
// and planes that touch the domain's ends ask where a value comes from a
// boundary rule (EDGE), and they write the boundary faces of u2 down, so that
// the drag reads faces alike everywhere;
// where the drag coefficient is zero (open air, most of a city) the face
// keeps its value, which is what the drag expression gives.  Measured at
// 256 x 256 x 64, FP32, against loops over the general expressions: 235 -> 137
// us (197 M -> 111 M warp instructions, issue slots 79 % busy), 512 x 512 x 128
// 1493 -> 737 us; the
// code of one variant more in the loop body cost 30 us in instruction fetch.
//
// Boundary faces of u~ and u2 are never stored between sub-steps; they come
// from the BC rules, as in the unfused kernels.
// Every value is formed by the expressions of k_diffuse, k_drag_bc and
// k_pressure_rhs; the blocks and z chunks are those of k_pressure_rhs
// (momentum_grid gives both), so ||b||^2 is summed in the same order.  The
// results, ||b||^2 included, are bit for bit those of the three kernels while
// the velocities are finite (in open air a face keeps its value here; the drag
// expression makes 0 of it beside an infinite one).
//
// Tape (the adjoint): when u2t is not null, u2 of every interior face the
// block owns is also written to (u2t, v2t, w2t).
#pragma once
#include "advect_fused.cuh"

namespace uf {

constexpr int DR = 4;   // ring of staged planes: k .. k+2 live, k+3 on its way
constexpr int UR = 2;   // ring of u2 planes
// staged fields, in this order, each [DR][MWP]
constexpr int DF_U = 0, DF_V = 1, DF_W = 2, DF_NUT = 3, DF_C = 4, DF_N = 5;
#ifndef UF_MOMENTUM_MINB
#define UF_MOMENTUM_MINB 4   // resident blocks per SM the register budget is sized for
#endif

template <typename T>
struct MomentumArgs {
  StepParams<T> p;
  const T* ut;
  const T* vt;
  const T* wt;       // advected velocity (interior faces)
  const T* nut;      // eddy viscosity (cells)
  const T* cc;       // drag coefficient (cells)
  T* u;
  T* v;
  T* w;              // out: u3 on every face
  T* b;              // out: right-hand side
  T* u2t;
  T* v2t;
  T* w2t;            // optional tape of u2 (interior faces)
  int zc;
  double* partials;
  SolveState* st;
};

template <typename T>
constexpr size_t momentum_fused_smem() {
  return sizeof(T) * ((size_t)DF_N * DR * MWP + (size_t)3 * UR * MHP + (size_t)(MX + 1) * MY + (size_t)MX * (MY + 1));
}

// One block's planes in its shared memory, as places (byte offsets).
template <typename T>
__device__ __forceinline__ T* mom_sm(int place) {
  extern __shared__ __align__(16) unsigned char mom_smem[];
  return reinterpret_cast<T*>(mom_smem + place);
}
template <typename T>
struct MView {
  static constexpr int B = sizeof(T);
  static constexpr int U2_0 = DF_N * DR * MWP, U3_0 = U2_0 + 3 * UR * MHP, V3_0 = U3_0 + (MX + 1) * MY;
  int i0, j0, k0, kend;
  __device__ __forceinline__ int D(int f, int k) const { return (f * DR + (k & (DR - 1))) * MWP * B; }     // plane k of staged field f
  __device__ __forceinline__ int U2(int q, int k) const { return (U2_0 + (q * UR + (k & 1)) * MHP) * B; }
  __device__ __forceinline__ T* sU3() const { return mom_sm<T>(U3_0 * B); }   // (MX+1) x MY: u3 of the plane's x faces
  __device__ __forceinline__ T* sV3() const { return mom_sm<T>(V3_0 * B); }   // MX x (MY+1): u3 of the plane's y faces
};

// Starts the copy of plane kk of the five staged fields into its ring slot
// (S: the thread's two window positions, stage_pos).
template <typename T>
__device__ __forceinline__ void stage_momentum(const MomentumArgs<T>& M, const MView<T>& V, const StagePos& S, int kk) {
  const StepParams<T>& p = M.p;
  if (kk < 0 || kk > p.nz) return;
  auto cell = [&](const T* at, const T* f) { return UF_PTR(at, f, p.Pc, p.ny, p.nz, 1, BA_CW); };
  T* dst = mom_sm<T>(V.D(0, kk)) + threadIdx.x;
  const size_t pc = (size_t)kk * ((size_t)p.Pc * p.ny);
  const T* su = M.ut + (size_t)kk * ((size_t)p.Pu * p.ny);
  const T* sv = M.vt + (size_t)kk * ((size_t)p.Pc * (p.ny + 1));
  const T *sw = M.wt + pc, *sn = M.nut + pc, *sc = M.cc + pc;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    T* d = dst + h * MT;
    if (kk < p.nz) {
      if (S.ok[h] & 1) cp_async_elem(d + DF_U * DR * MWP, UF_PTR(su + S.u[h], M.ut, p.Pu, p.ny, p.nz, 1, BA_U));
      if (S.ok[h] & 2) cp_async_elem(d + DF_V * DR * MWP, UF_PTR(sv + S.c[h], M.vt, p.Pc, p.ny + 1, p.nz, 1, BA_V));
      if (S.ok[h] & 4) {
        cp_async_elem(d + DF_NUT * DR * MWP, cell(sn + S.c[h], M.nut));
        cp_async_elem(d + DF_C * DR * MWP, cell(sc + S.c[h], M.cc));
      }
    }
    if (S.ok[h] & 4) cp_async_elem(d + DF_W * DR * MWP, UF_PTR(sw + S.c[h], M.wt, p.Pc, p.ny, p.nz + 1, 1, BA_CW));
  }
}

// Diffusion of one interior face (the expressions of diffuse_body) from its
// six neighbours.
template <typename T>
__device__ __forceinline__ T diffuse_face(const StepParams<T>& p, T c, T x0, T xm, T xp, T ym, T yp, T zm, T zp, T n0, T n1) {
  const T lap = xm + xp + ym + yp + zm + zp - T(6) * x0;
  const T nf = T(0.5) * (n0 + n1);
  return x0 + c * (p.nu + nf) * lap;
}
// ... of a face with all its neighbours inside; f: its place in the plane.
template <typename T>
__device__ __forceinline__ T diffuse_inner(const StepParams<T>& p, T c, const T* f, T x0, T zm, T zp, T n0, T n1) {
  return diffuse_face(p, c, x0, f[-1], f[1], f[-MWX], f[MWX], zm, zp, n0, n1);
}
// u2 of component Q at lattice point (i, j, m) near the domain's ends, b its
// place in the staged window; in: the component's inflow value of the plane.
// A boundary face takes its rule's value (at an outlet that of the adjacent
// interior face, formed here too), so that whoever reads u2 finds every face.
// 0 off the lattice.
template <int Q, typename T>
__device__ __forceinline__ T u2_edge(const StepParams<T>& p, const MView<T>& V, T c, int b, int i, int j, int m, T in) {
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  if (i < 0 || j < 0 || m < 0 || i >= nx + (Q == 0) || j >= ny + (Q == 1) || m >= nz + (Q == 2)) return T(0);
  if (Q == 2 && (m == 0 || m == nz)) return T(0);
  int rule = NOSLIP + 1;   // of a boundary face
  if (Q == 0) {
    if (i == 0) { rule = p.side[0]; i += 1; b += 1; }
    else if (i == nx) { rule = p.side[1]; i -= 1; b -= 1; }
  }
  if (Q == 1) {
    if (j == 0) { rule = p.side[2]; j += 1; b += MWX; }
    else if (j == ny) { rule = p.side[3]; j -= 1; b -= MWX; }
  }
  const T *f = mom_sm<T>(V.D(Q, m)) + b, *n = mom_sm<T>(V.D(DF_NUT, m)) + b;
  const T x0 = f[0];
  T xm = f[-1], xp = f[1], ym = f[-MWX], yp = f[MWX], zm = mom_sm<T>(V.D(Q, m - 1))[b], zp = mom_sm<T>(V.D(Q, m + 1))[b];
  // along its own axis the neighbour may be a boundary face, along the others a ghost
  if (Q == 0) {
    if (i == 1) xm = normal_face(p.side[0], x0, in);
    if (i == nx - 1) xp = normal_face(p.side[1], x0, in);
  } else {
    if (i == 0) xm = tangential_ghost(p.side[0], x0, in);
    if (i == nx - 1) xp = tangential_ghost(p.side[1], x0, in);
  }
  if (Q == 1) {
    if (j == 1) ym = normal_face(p.side[2], x0, in);
    if (j == ny - 1) yp = normal_face(p.side[3], x0, in);
  } else {
    if (j == 0) ym = tangential_ghost(p.side[2], x0, in);
    if (j == ny - 1) yp = tangential_ghost(p.side[3], x0, in);
  }
  if (Q == 2) {
    if (m == 1) zm = T(0);
    if (m == nz - 1) zp = T(0);
  } else {
    if (m == 0) zm = tangential_ghost(p.side[4], x0, T(0));
    if (m == nz - 1) zp = tangential_ghost(p.side[5], x0, T(0));
  }
  const T n0 = Q == 0 ? n[-1] : (Q == 1 ? n[-MWX] : mom_sm<T>(V.D(DF_NUT, m - 1))[b]);
  const T val = diffuse_face(p, c, x0, xm, xp, ym, yp, zm, zp, n0, n[0]);
  return rule > NOSLIP ? val : normal_face(rule, val, in);
}
template <int Q, typename T>
__device__ __forceinline__ void tape_u2(const MomentumArgs<T>& M, const MView<T>& V, int i, int j, int m, T val) {
  // the column's own interior faces
  if (m < V.k0 || m >= V.kend || i >= M.p.nx || j >= M.p.ny || (Q == 0 ? i : (Q == 1 ? j : m)) == 0) return;
  if (Q == 0) M.u2t[idx_u(M.p, i, j, m)] = val;
  else if (Q == 1) M.v2t[idx_v(M.p, i, j, m)] = val;
  else M.w2t[idx_c(M.p, i, j, m)] = val;
}

// A thread's own staged values on the planes m - 1 and m (u~, v~, w~, nu_t),
// rolled along the march.
template <typename T>
struct OwnColumn {
  T below[4], here[4];
  __device__ __forceinline__ void start(const MView<T>& V, int b, int m) {   // before u2_plane(m)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      below[f] = mom_sm<T>(V.D(f, m - 1))[b];
      here[f] = mom_sm<T>(V.D(f, m))[b];
    }
  }
};

// u2 on plane m: the thread's own faces and its halo face.
template <bool EDGE, typename T>
__device__ __forceinline__ void u2_plane(const MomentumArgs<T>& M, const MView<T>& V, const Places& X, OwnColumn<T>& O, T c, int m) {
  const StepParams<T>& p = M.p;
  constexpr int FS = DR * MWP, US = UR * MHP;   // from one field (component) to the next
  const T* fc = mom_sm<T>(V.D(0, m)) + X.b;
  const T* fp = mom_sm<T>(V.D(0, m + 1)) + X.b;
  T* u2 = mom_sm<T>(V.U2(0, m));
  T next[4];
#pragma unroll
  for (int f = 0; f < 4; ++f) next[f] = fp[f * FS];
  if (EDGE) {
    const T prof = m >= 0 && m < p.nz ? p.prof[m] : T(0);
    const T inu = prof * p.dirx, inv = prof * p.diry;
    const T a = u2_edge<0>(p, V, c, X.b, X.gi, X.gj, m, inu);
    const T b = u2_edge<1>(p, V, c, X.b, X.gi, X.gj, m, inv);
    const T w = u2_edge<2>(p, V, c, X.b, X.gi, X.gj, m, T(0));
    T h = 0;
    if (X.hq == 0) h = u2_edge<0>(p, V, c, X.hb, X.hi, X.hj, m, inu);
    else if (X.hq == 1) h = u2_edge<1>(p, V, c, X.hb, X.hi, X.hj, m, inv);
    else if (X.hq == 2) h = u2_edge<2>(p, V, c, X.hb, X.hi, X.hj, m, T(0));
    u2[X.h] = a;
    u2[US + X.h] = b;
    u2[2 * US + X.h] = w;
    if (X.hq < 3) u2[X.hq * US + X.hh] = h;
    if (M.u2t) {
      tape_u2<0>(M, V, X.gi, X.gj, m, a);
      tape_u2<1>(M, V, X.gi, X.gj, m, b);
      tape_u2<2>(M, V, X.gi, X.gj, m, w);
    }
  } else {
    const T* n = fc + 3 * FS;
    const T a = diffuse_inner(p, c, fc, O.here[0], O.below[0], next[0], n[-1], O.here[3]);
    const T b = diffuse_inner(p, c, fc + FS, O.here[1], O.below[1], next[1], n[-MWX], O.here[3]);
    const T w = diffuse_inner(p, c, fc + 2 * FS, O.here[2], O.below[2], next[2], O.below[3], O.here[3]);
    T h = 0;
    if (X.hq < 3) {
      const T* g = mom_sm<T>(V.D(0, m)) + X.hq * FS + X.hb;
      const T *gm = mom_sm<T>(V.D(0, m - 1)) + X.hb, *gp = mom_sm<T>(V.D(0, m + 1)) + X.hb;
      const T* gn = mom_sm<T>(V.D(DF_NUT, m)) + X.hb;
      h = diffuse_inner(p, c, g, g[0], gm[X.hq * FS], gp[X.hq * FS], X.hq == 2 ? gm[3 * FS] : gn[X.hq == 0 ? -1 : -MWX], gn[0]);
    }
    u2[X.h] = a;
    u2[US + X.h] = b;
    u2[2 * US + X.h] = w;
    if (X.hq < 3) u2[X.hq * US + X.hh] = h;
    if (M.u2t) {
      tape_u2<0>(M, V, X.gi, X.gj, m, a);
      tape_u2<1>(M, V, X.gi, X.gj, m, b);
      tape_u2<2>(M, V, X.gi, X.gj, m, w);
    }
  }
#pragma unroll
  for (int f = 0; f < 4; ++f) {
    O.below[f] = O.here[f];
    O.here[f] = next[f];
  }
}

// Drag of a face away from the domain's ends: q its value, cf the mean drag
// coefficient, a0..a3 and b0..b3 the four faces around it of the other two
// components, in the order of drag_at; o: its position among q and the two
// means (0, 1, 2 for u, v, w).  With cf = 0 the factor is exactly 1.
template <int O, typename T, typename FA, typename FB>
__device__ __forceinline__ T drag_inner(T dt, T q, T cf, FA a, FB b) {
  if (cf == T(0)) return q;
  const T am = T(0.25) * (a(0) + a(1) + a(2) + a(3));
  const T bm = T(0.25) * (b(0) + b(1) + b(2) + b(3));
  const T sp = O == 0 ? sqrt(q * q + am * am + bm * bm) : (O == 1 ? sqrt(am * am + q * q + bm * bm) : sqrt(am * am + bm * bm + q * q));
  return fmax(T(0), T(1) - dt * cf * sp) * q;
}
// u3 of a face away from the ends at places h (u2 window) and s (staged
// window): an x face and a y face of plane k, a z face of plane k.
template <typename T>
__device__ __forceinline__ T u3_inner(const MView<T>& V, T dt, int h, int s, int k) {
  const T *u = mom_sm<T>(V.U2(0, k)) + h, *v = mom_sm<T>(V.U2(1, k)) + h, *w = mom_sm<T>(V.U2(2, k)) + h, *wp = mom_sm<T>(V.U2(2, k + 1)) + h;
  const T* C = mom_sm<T>(V.D(DF_C, k)) + s;
  return drag_inner<0>(dt, u[0], T(0.5) * (C[-1] + C[0]), [&](int e) { return v[-1 + (e & 1) + (e >> 1) * MHX]; },
                       [&](int e) { return (e < 2 ? w : wp)[-1 + (e & 1)]; });
}
template <typename T>
__device__ __forceinline__ T v3_inner(const MView<T>& V, T dt, int h, int s, int k) {
  const T *u = mom_sm<T>(V.U2(0, k)) + h, *v = mom_sm<T>(V.U2(1, k)) + h, *w = mom_sm<T>(V.U2(2, k)) + h, *wp = mom_sm<T>(V.U2(2, k + 1)) + h;
  const T* C = mom_sm<T>(V.D(DF_C, k)) + s;
  return drag_inner<1>(dt, v[0], T(0.5) * (C[-MWX] + C[0]), [&](int e) { return u[-MHX + (e & 1) + (e >> 1) * MHX]; },
                       [&](int e) { return (e < 2 ? w : wp)[-MHX + (e & 1) * MHX]; });
}
template <typename T>
__device__ __forceinline__ T w3_inner(const MView<T>& V, T dt, int h, int s, int k) {
  const T *u = mom_sm<T>(V.U2(0, k)) + h, *v = mom_sm<T>(V.U2(1, k)) + h, *w = mom_sm<T>(V.U2(2, k)) + h;
  const T *um = mom_sm<T>(V.U2(0, k - 1)) + h, *vm = mom_sm<T>(V.U2(1, k - 1)) + h;
  const T c0 = mom_sm<T>(V.D(DF_C, k - 1))[s], c1 = mom_sm<T>(V.D(DF_C, k))[s];
  return drag_inner<2>(dt, w[0], T(0.5) * (c0 + c1), [&](int e) { return (e < 2 ? um : u)[e & 1]; },
                       [&](int e) { return (e < 2 ? vm : v)[(e & 1) * MHX]; });
}

// u3 on the faces of plane k and the w faces of plane k + 1 (only_w: those
// alone); the x and y faces go to shared memory for the fluxes.  own[]: the
// thread's own u3, v3 of plane k and w3 of plane k + 1.  The faces on the
// column's far sides, the row j0 + MY of y faces and the column i0 + MX of x
// faces, are formed by the first warp and by a lane per row of the second.
template <bool EDGE, typename T>
__device__ __forceinline__ void u3_plane(const MomentumArgs<T>& M, const MView<T>& V, const Places& X, T dt, int k, bool only_w,
                                         T (&own)[3]) {
  const StepParams<T>& p = M.p;
  const int t = threadIdx.x, tx = t % MX, ty = t / MX;
  T *sU = V.sU3(), *sV = V.sV3();
  T* gu = M.u + (size_t)k * ((size_t)p.Pu * p.ny);
  T* gv = M.v + (size_t)k * ((size_t)p.Pc * (p.ny + 1));
  T* gw = M.w + (size_t)(k + 1) * ((size_t)p.Pc * p.ny);
  auto U = [&](T* at) { return UF_PTR(at, M.u, p.Pu, p.ny, p.nz, 1, BA_U); };
  auto VV = [&](T* at) { return UF_PTR(at, M.v, p.Pc, p.ny + 1, p.nz, 1, BA_V); };
  const bool own_w = k + 1 < V.kend || k + 1 == p.nz;
  const T prof = EDGE && k >= 0 ? p.prof[k] : T(0);
  // x face (i, j) and y face (i, j): places h, b; a boundary face follows its rule on the dragged interior neighbour
  auto xface = [&](int h, int b, int i) {
    const int sh = EDGE ? (i == 0 ? 1 : (i == p.nx ? -1 : 0)) : 0;
    const T r = u3_inner(V, dt, h + sh, b + sh, k);
    return EDGE && sh ? normal_face(p.side[i == 0 ? 0 : 1], r, prof * p.dirx) : r;
  };
  auto yface = [&](int h, int b, int j) {
    const int sh = EDGE ? (j == 0 ? 1 : (j == p.ny ? -1 : 0)) : 0;
    const T r = v3_inner(V, dt, h + sh * MHX, b + sh * MWX, k);
    return EDGE && sh ? normal_face(p.side[j == 0 ? 2 : 3], r, prof * p.diry) : r;
  };
  const int gi = X.gi, gj = X.gj;
  const bool in_x = !EDGE || gi < p.nx, in_y = !EDGE || gj < p.ny;
  if (in_x && in_y) {
    own[2] = EDGE && (k + 1 == 0 || k + 1 == p.nz) ? T(0) : w3_inner(V, dt, X.h, X.b, k + 1);
    if (own_w) *UF_PTR(gw + (gi + p.Pc * gj), M.w, p.Pc, p.ny, p.nz + 1, 1, BA_CW) = own[2];
  }
  if (only_w) return;
  if (!EDGE || (gi <= p.nx && in_y)) {
    own[0] = xface(X.h, X.b, gi);
    sU[tx + (MX + 1) * ty] = own[0];
    *U(gu + (gi + p.Pu * gj)) = own[0];
  }
  if (!EDGE || (in_x && gj <= p.ny)) {
    own[1] = yface(X.h, X.b, gj);
    sV[t] = own[1];
    *VV(gv + (gi + p.Pc * gj)) = own[1];
  }
  if (t < MX) {
    const int j = V.j0 + MY;
    if (!EDGE || (in_x && j <= p.ny)) {
      const T val = yface(X.h + MHX * MY, X.b + MWX * MY, j);
      sV[t + MT] = val;
      if (EDGE && j == p.ny) *VV(gv + (gi + p.Pc * j)) = val;
    }
  } else if (t < MX + MY) {
    const int i = V.i0 + MX, j = V.j0 + tx;
    if (!EDGE || (i <= p.nx && j < p.ny)) {
      const T val = xface(MX + 1 + MHX * (tx + 1), MX + 2 + MWX * (tx + 2), i);
      sU[MX + (MX + 1) * tx] = val;
      if (EDGE && i == p.nx) *U(gu + (i + p.Pu * j)) = val;
    }
  }
}

template <typename T>
__device__ __forceinline__ void momentum_fused_body(const MomentumArgs<T>& M, const VBlock& vb) {
  __shared__ double sh[32];
  __shared__ bool last;
  const StepParams<T>& p = M.p;
  MView<T> V;
  V.i0 = vb.x * MX;
  V.j0 = vb.y * MY;
  V.k0 = vb.z * M.zc;
  V.kend = min(p.nz, V.k0 + M.zc);
  const int k0 = V.k0, kend = V.kend;
  const int tx = threadIdx.x % MX, ty = threadIdx.x / MX;
  const Places X = block_places(V.i0, V.j0);
  const bool own_c = X.gi < p.nx && X.gj < p.ny;
  const T dt = *p.dtT;
  const T c = dt * p.inv_h * p.inv_h;
  const T sc = -p.rho * p.h / *p.dtT;
  StagePos S;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t = threadIdx.x + h * MT, gx = V.i0 - 2 + t % MWX, gy = V.j0 - 2 + t / MWX;
    const bool in = t < MWP && gx >= 0 && gy >= 0;
    S.u[h] = gx + p.Pu * gy;
    S.c[h] = gx + p.Pc * gy;
    S.ok[h] = !in ? 0 : (gx <= p.nx && gy < p.ny ? 1 : 0) | (gx < p.nx && gy <= p.ny ? 2 : 0) | (gx < p.nx && gy < p.ny ? 4 : 0);
  }
  // no face of the halo-1 window, nor a neighbour of one, on the domain's x and y ends
  const bool inner = V.i0 >= 3 && V.i0 + MX + 1 <= p.nx - 1 && V.j0 >= 3 && V.j0 + MY + 1 <= p.ny - 1;
  auto edge2 = [&](int m) { return !inner || m < 2 || m > p.nz - 2; };          // of u2 on plane m
  auto edge3 = [&](int k) { return !inner || k < 1 || k + 1 > p.nz - 1; };      // of u3 on plane k and w3 on k + 1
  for (int kk = k0 - 2; kk <= k0; ++kk) stage_momentum(M, V, S, kk);
  cp_async_commit();
  DotAcc<T> dacc;
  T own[3] = {T(0), T(0), T(0)}, w3lo = T(0);
  OwnColumn<T> O;
  // b of plane k from the faces in shared memory and the thread's own
  auto rhs = [&](int k) {
    // cell_flux: u(i+1)-u(i) + v(j+1)-v(j) + w(k+1)-w(k)
    const T flux = V.sU3()[(tx + 1) + (MX + 1) * ty] - own[0] + V.sV3()[tx + MX * (ty + 1)] - own[1] + own[2] - w3lo;
    const T bv = sc * flux;
    *UF_PTR(M.b + (size_t)k * ((size_t)p.Pc * p.ny) + (X.gi + p.Pc * X.gj), M.b, p.Pc, p.ny, p.nz, 1, BA_CW) = bv;
    dacc.add(bv, bv);
    w3lo = own[2];
  };
  // m: the plane of u2; the faces follow one plane behind, b another one
  for (int m = k0 - 1; m <= kend; ++m) {
    const int k = m - 1;
    cp_async_wait_all();
    __syncthreads();
    stage_momentum(M, V, S, m + 2);   // into the slot of m - 2
    cp_async_commit();
    if (m == k0 - 1) O.start(V, X.b, m);
    if (k > k0 && own_c) rhs(k - 1);
    if (edge2(m)) u2_plane<true>(M, V, X, O, c, m);
    else u2_plane<false>(M, V, X, O, c, m);
    if (m < k0) continue;
    __syncthreads();
    // (at m = k0 only the w faces of the column's bottom, for the first flux)
    if (edge3(k)) u3_plane<true>(M, V, X, dt, k, k < k0, own);
    else u3_plane<false>(M, V, X, dt, k, k < k0, own);
    if (k < k0) w3lo = own[2];
  }
  __syncthreads();
  if (own_c) rhs(kend - 1);
  cp_async_wait_all();
  double acc = 0.0;
  acc += dacc.value();
  acc = block_sum<NT>(acc, sh);
  const double vals[1] = {acc};
  if (publish_partials<1>(M.partials, &M.st->ticket[0], vals, &last, vb)) {
    double tot[1];
    reduce_partials_sum<NT, 1>(M.partials, tot, sh, vb.n);
    if (thread_linear_id() == 0) {
      M.st->bb = tot[0];
      M.st->iter = 0;
      M.st->converged = 0;
      M.st->status = DEV_OK;
      M.st->ticket[0] = 0u;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(MT, sizeof(T) == 8 ? 2 : UF_MOMENTUM_MINB) k_momentum_fused(const __grid_constant__ MomentumArgs<T> M) {
  momentum_fused_body<T>(M, vblock());
}

}  // namespace uf
