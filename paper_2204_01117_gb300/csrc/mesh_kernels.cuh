// Mesh resolver of Sec. 3 ("Urban model resolving"): cell porosity from
// closed triangle meshes.  A point is inside an object when it lies in the
// object's axis-aligned bounding box and a ray from it crosses the object's
// triangles an odd number of times (even-odd rule); crossings by the
// Moller-Trumbore test (1997), here without the division by the
// determinant: the barycentric and distance tests compare against |det|.
// A cell's porosity is the mean over a uniform sub-grid of sub^3 points of
// the minimum inside porosity of the objects containing the point (1 in the
// open), the volume fraction outside the solids of the cut-cell treatment.
// A point's classification is integer work decided by floating point, so
// every product and sum is a separate round-to-nearest FP64 operation in a
// fixed order (the _rn intrinsics are never fused into FMAs).
#pragma once
#include <cuda_runtime.h>

#include "uf_device.cuh"

namespace uf {

// Ray direction: no zero component, so no face of an axis-aligned box is
// parallel to it.
constexpr double RAY_X = 0.5741, RAY_Y = 0.6219, RAY_Z = 0.5327;

struct MeshObject {
  int first, count;     // triangles [first, first + count)
  double phi_in;        // porosity inside
  double lo[3], hi[3];  // bounding box [m]
  int clo[3], chi[3];   // cells [clo, chi] per axis whose closed box meets the bounding box
  int entry;            // its triangles' first entry in the tables below
  double scale;         // 1 / (size of the bounding box + 2 h): local coordinates (p - lo) scale lie in about [0, 1]
};

// What the crossing test needs of a triangle whatever the point: the edges,
// q = RAY x e2, the determinant's sign and size (0: parallel to the ray), each
// formed as the test forms them.
struct MeshTri {
  double v0[3], e1[3], e2[3], q[3], s, adet;
};
// The same test in FP32 in the object's local coordinates.  u, w and t of the
// test are affine in the point: f(p) = a . (p - v0); e bounds the rounding of
// f, in FP32 here and in FP64 there: 2e-6 sum |a| (32 units in the last place
// of local coordinates, coefficients and sums), and 2e-6 of the determinant.
struct MeshTriF {
  float v[3], adet;     // adet < 0: the ray never crosses
  float u[3], eu;
  float w[3], ew;
  float t[3], et;
};

__device__ __forceinline__ double dot3_rn(double ax, double ay, double az, double bx, double by, double bz) {
  return __dadd_rn(__dadd_rn(__dmul_rn(ax, bx), __dmul_rn(ay, by)), __dmul_rn(az, bz));
}

__device__ __forceinline__ double mesh_tri(const double* v, MeshTri& o) {   // the determinant
  for (int a = 0; a < 3; ++a) {
    o.v0[a] = v[a];
    o.e1[a] = __dsub_rn(v[3 + a], v[a]);
    o.e2[a] = __dsub_rn(v[6 + a], v[a]);
  }
  // q = RAY x e2, det = e1 . q
  o.q[0] = __dsub_rn(__dmul_rn(RAY_Y, o.e2[2]), __dmul_rn(RAY_Z, o.e2[1]));
  o.q[1] = __dsub_rn(__dmul_rn(RAY_Z, o.e2[0]), __dmul_rn(RAY_X, o.e2[2]));
  o.q[2] = __dsub_rn(__dmul_rn(RAY_X, o.e2[1]), __dmul_rn(RAY_Y, o.e2[0]));
  const double det = dot3_rn(o.e1[0], o.e1[1], o.e1[2], o.q[0], o.q[1], o.q[2]);
  o.s = det > 0.0 ? 1.0 : -1.0;
  o.adet = det == 0.0 ? 0.0 : __dmul_rn(det, o.s);
  return det;
}
// Fills an object's table entries (one block per object).
__device__ __forceinline__ void mesh_prep_tri(const double* v, const MeshObject& m, MeshTri& o, MeshTriF& f) {
  const double det = mesh_tri(v, o);
  const double c = m.scale, c2 = c * c, g = o.s;
  // w = RAY . (p x e1) = p . (e1 x RAY), t = e2 . (p x e1) = p . (e1 x e2)
  const double w[3] = {o.e1[1] * RAY_Z - o.e1[2] * RAY_Y, o.e1[2] * RAY_X - o.e1[0] * RAY_Z, o.e1[0] * RAY_Y - o.e1[1] * RAY_X};
  const double t[3] = {o.e1[1] * o.e2[2] - o.e1[2] * o.e2[1], o.e1[2] * o.e2[0] - o.e1[0] * o.e2[2],
                       o.e1[0] * o.e2[1] - o.e1[1] * o.e2[0]};
  float su = 0.f, sw = 0.f, st = 0.f;
  for (int a = 0; a < 3; ++a) {
    f.v[a] = (float)((v[a] - m.lo[a]) * c);
    f.u[a] = (float)(g * o.q[a] * c);
    f.w[a] = (float)(g * w[a] * c);
    f.t[a] = (float)(g * t[a] * c2);
    su += fabsf(f.u[a]);
    sw += fabsf(f.w[a]);
    st += fabsf(f.t[a]);
  }
  f.adet = det == 0.0 ? -1.f : (float)(o.adet * c2);
  const float e0 = 1e-30f + 2e-6f * fabsf(f.adet);
  f.eu = 2e-6f * su + e0;
  f.ew = 2e-6f * sw + e0;
  f.et = 2e-6f * st + e0;
}
template <int NT_>
__global__ void __launch_bounds__(NT_) k_mesh_prep(const double* __restrict__ tri, const MeshObject* __restrict__ obj, MeshTri* te,
                                                   MeshTriF* tf) {
  const MeshObject m = obj[blockIdx.x];
  for (int e = threadIdx.x; e < m.count; e += NT_) mesh_prep_tri(tri + 9 * ((size_t)m.first + e), m, te[m.entry + e], tf[m.entry + e]);
}

// Whether the ray p + t RAY, t > 0, crosses the triangle: the test itself.
__device__ __forceinline__ bool ray_crosses(double px, double py, double pz, const MeshTri& o) {
  const double tx = __dsub_rn(px, o.v0[0]), ty = __dsub_rn(py, o.v0[1]), tz = __dsub_rn(pz, o.v0[2]);
  const double u = __dmul_rn(dot3_rn(tx, ty, tz, o.q[0], o.q[1], o.q[2]), o.s);
  // r = t x e1
  const double rx = __dsub_rn(__dmul_rn(ty, o.e1[2]), __dmul_rn(tz, o.e1[1]));
  const double ry = __dsub_rn(__dmul_rn(tz, o.e1[0]), __dmul_rn(tx, o.e1[2]));
  const double rz = __dsub_rn(__dmul_rn(tx, o.e1[1]), __dmul_rn(ty, o.e1[0]));
  const double w = __dmul_rn(dot3_rn(RAY_X, RAY_Y, RAY_Z, rx, ry, rz), o.s);
  const double t = __dmul_rn(dot3_rn(o.e2[0], o.e2[1], o.e2[2], rx, ry, rz), o.s);
  return u >= 0.0 && u <= o.adet && w >= 0.0 && __dadd_rn(u, w) <= o.adet && t > 0.0;
}
// The same for every point within r (local, per axis) of the local point p:
// -1 none of them crosses, 1 all of them do, 0 the FP32 bounds cannot tell.
__device__ __forceinline__ int ray_bound(float px, float py, float pz, float r, const MeshTriF& f) {
  if (f.adet < 0.f) return -1;
  const float dx = px - f.v[0], dy = py - f.v[1], dz = pz - f.v[2];
  const float u = f.u[0] * dx + f.u[1] * dy + f.u[2] * dz, w = f.w[0] * dx + f.w[1] * dy + f.w[2] * dz;
  const float t = f.t[0] * dx + f.t[1] * dy + f.t[2] * dz, a = f.adet;
  const float eu = f.eu + r * (fabsf(f.u[0]) + fabsf(f.u[1]) + fabsf(f.u[2]));
  const float ew = f.ew + r * (fabsf(f.w[0]) + fabsf(f.w[1]) + fabsf(f.w[2]));
  const float et = f.et + r * (fabsf(f.t[0]) + fabsf(f.t[1]) + fabsf(f.t[2]));
  const float eb = f.eu + f.ew + r * (fabsf(f.u[0] + f.w[0]) + fabsf(f.u[1] + f.w[1]) + fabsf(f.u[2] + f.w[2]));
  if (u < -eu || u - a > eu || w < -ew || u + w - a > eb || t < -et) return -1;
  if (u > eu && a - u > eu && w > ew && a - u - w > eb && t > et) return 1;
  return 0;
}

// A block takes a brick of cells, a warp one to 32 of them: the brick's objects
// are listed once (a brick in the open, most of a city, is 1 at once), then
// each warp works through those of its cells that an object's cell range
// holds.  For such a cell the lanes list its objects and bound every triangle of
// each over the whole cell: a triangle that no ray from the cell can cross drops
// out, one that every ray crosses only flips the parity, the few others are
// listed.  The sub^3 sample points, 32 at a time, then test the listed ones,
// in FP32 where its bound decides and with the test itself where it does not.
// Every decision is the test's, so the field is the same bit for bit; what
// bounded the kernel before were FP64 tests of every point against every
// triangle (1/64 rate) and the serial object list of every cell.  Measured at
// 256 x 256 x 64 with 100 objects (6500 triangles), the whole call: 23.4 ->
// 1.07 ms.
// The brick: 8 x 8 x 4 cells, 32 to a warp, while the grid has cells for about
// 32 warps on each SM, halved until it has, down to a cell to a warp: on a
// coarse grid, whose cells hold many objects each, a warp would work through
// its cells one after another while most of the chip had none (12 x 12 x 4 with
// 300 objects 1.7 ms against 13.8, 50 x 50 x 8 with 4000 11 against
// 114, also for the lists of 64 objects to a brick, past which every point met every
// object).
// TABLES = false: a mesh whose tables do not fit (an entry per object and
// triangle, so objects that share long ranges need many) is tested triangle
// by triangle.
constexpr int MESH_BRICK = 1024;   // objects of a brick (more: its cells look through all)
constexpr int MESH_LIST = 64;      // objects of a cell (more: every point visits the brick's)
constexpr int MESH_OPEN = 192;     // undecided triangles of a cell (more: every triangle is tested)
constexpr int MESH_WARPS = 8;
// Brick of 2^(x + y + z) cells, 2^(x + y + z - 3) to a warp.
struct MeshBrick {
  int x, y, z;
};
inline MeshBrick mesh_brick(int nx, int ny, int nz) {
  const MeshBrick bricks[] = {{3, 3, 2}, {3, 2, 2}, {2, 2, 2}, {2, 2, 1}, {2, 1, 1}};
  for (const MeshBrick& b : bricks)
    if (((size_t)nx * ny * nz >> (b.x + b.y + b.z - 3)) >= 152 * 32) return b;
  return {1, 1, 1};
}
inline unsigned mesh_blocks(int nx, int ny, int nz, MeshBrick b) {   // bricks, x fastest (in one dimension: any nz)
  return (unsigned)((size_t)((nx + (1 << b.x) - 1) >> b.x) * ((ny + (1 << b.y) - 1) >> b.y) * ((nz + (1 << b.z) - 1) >> b.z));
}
template <typename T, bool TABLES>
__global__ void __launch_bounds__(32 * MESH_WARPS) k_mesh_phi(int nx, int ny, int nz, int P, double h, int sub, MeshBrick brick,
                                                              const double* __restrict__ tri, const MeshTri* __restrict__ te,
                                                              const MeshTriF* __restrict__ tf, const MeshObject* __restrict__ obj,
                                                              int nobj, T* __restrict__ phi) {
  __shared__ int s_obj[MESH_BRICK], s_nobj;
  __shared__ int s_cell[MESH_WARPS][MESH_LIST];          // objects of the warp's cell
  __shared__ int s_open[MESH_WARPS][MESH_OPEN];          // its undecided triangles, object by object
  __shared__ int s_end[MESH_WARPS][MESH_LIST];           // where each object's end
  __shared__ unsigned char s_odd[MESH_WARPS][MESH_LIST]; // parity of the crossings common to the whole cell
  __shared__ double s_val[MESH_WARPS][32];
  __shared__ double s_off[16];          // sample offsets (a + 1/2) / sub within a cell
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const unsigned int nbx = (nx + (1 << brick.x) - 1) >> brick.x, nby = (ny + (1 << brick.y) - 1) >> brick.y, row = blockIdx.x / nbx;
  const int bi = (int)(blockIdx.x % nbx) << brick.x, bj = (int)(row % nby) << brick.y, bk = (int)(row / nby) << brick.z;
  if (t == 0) s_nobj = 0;
  if (t < sub) s_off[t] = __ddiv_rn(__dadd_rn((double)t, 0.5), (double)sub);
  __syncthreads();
  for (int o = t; o < nobj; o += 32 * MESH_WARPS) {
    const MeshObject& m = obj[o];
    if (bi + (1 << brick.x) - 1 < m.clo[0] || bi > m.chi[0] || bj + (1 << brick.y) - 1 < m.clo[1] || bj > m.chi[1] ||
        bk + (1 << brick.z) - 1 < m.clo[2] || bk > m.chi[2])
      continue;
    const int at = atomicAdd(&s_nobj, 1);
    if (at < MESH_BRICK) s_obj[at] = o;
  }
  __syncthreads();
  const bool all = s_nobj > MESH_BRICK;              // too many: look through every object
  const int n_obj = all ? nobj : s_nobj;
  const int per_warp = 1 << (brick.x + brick.y + brick.z - 3), cell = warp * per_warp + lane;
  const int i = bi + (cell & ((1 << brick.x) - 1)), j = bj + (cell >> brick.x & ((1 << brick.y) - 1)), k = bk + (cell >> (brick.x + brick.y));
  const bool in = lane < per_warp && i < nx && j < ny && k < nz;
  auto holds = [&](const MeshObject& m, int a, int b, int c) {
    return a >= m.clo[0] && a <= m.chi[0] && b >= m.clo[1] && b <= m.chi[1] && c >= m.clo[2] && c <= m.chi[2];
  };
  bool hit = n_obj > MESH_LIST;                      // (then the cells' lists tell)
  for (int q = 0; q < n_obj && !hit; ++q) hit = holds(obj[s_obj[q]], i, j, k);
  T out = T(1);                                      // the open: every point is 1, and so is their mean
  const int npts = sub * sub * sub;
  const double hh = 0.5 * h;
  for (unsigned int todo = __ballot_sync(0xffffffffu, in && hit); todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1;
    const int ci = __shfl_sync(0xffffffffu, i, src), cj = __shfl_sync(0xffffffffu, j, src), ck = __shfl_sync(0xffffffffu, k, src);
    // list the cell's objects
    int nl = 0;
    for (int q = 0; q < n_obj; q += 32) {
      const int o = q + lane < n_obj ? (all ? q + lane : s_obj[q + lane]) : -1;
      const bool has = o >= 0 && holds(obj[o], ci, cj, ck);
      const unsigned int m = __ballot_sync(0xffffffffu, has);
      const int at = nl + __popc(m & ((1u << lane) - 1u));
      if (has && at < MESH_LIST) s_cell[warp][at] = o;
      nl += __popc(m);
    }
    if (nl == 0) continue;
    const bool over = nl > MESH_LIST;                // too many: every point visits the brick's
    __syncwarp();
    // bound the triangles over the cell
    bool exact = !TABLES || over;                    // too much to list: test every triangle
    int n = 0;
    for (int q = 0; q < nl && !exact; ++q) {
      const MeshObject& m = obj[s_cell[warp][q]];
      unsigned int odd = 0;
      const float px = (float)(((ci + 0.5) * h - m.lo[0]) * m.scale), py = (float)(((cj + 0.5) * h - m.lo[1]) * m.scale),
                  pz = (float)(((ck + 0.5) * h - m.lo[2]) * m.scale), r = (float)(hh * m.scale) * 1.0001f;
      for (int e = 0; e < m.count; e += 32) {
        int b = -1;
        if (e + lane < m.count) b = ray_bound(px, py, pz, r, tf[m.entry + e + lane]);
        odd ^= __popc(__ballot_sync(0xffffffffu, b == 1)) & 1u;
        const unsigned int open = __ballot_sync(0xffffffffu, b == 0);
        const int at = n + __popc(open & ((1u << lane) - 1u));
        if (b == 0 && at < MESH_OPEN) s_open[warp][at] = m.entry + e + lane;
        n += __popc(open);
      }
      if (n > MESH_OPEN) exact = true;
      if (lane == 0) {
        s_end[warp][q] = n;
        s_odd[warp][q] = (unsigned char)odd;
      }
    }
    __syncwarp();
    double acc = 0.0;
    bool whole = true;                               // acc is a whole number: the order of its sum does not matter
    for (int base = 0; base < npts; base += 32) {
      const int e = base + lane;
      double val = 1.0;
      const int a = e % sub, b = (e / sub) % sub, c = e / (sub * sub);
      const bool pt = e < npts;
      const double px = __dmul_rn(__dadd_rn((double)ci, s_off[pt ? a : 0]), h);
      const double py = __dmul_rn(__dadd_rn((double)cj, s_off[pt ? b : 0]), h);
      const double pz = __dmul_rn(__dadd_rn((double)ck, s_off[pt ? c : 0]), h);
      for (int q = 0, at = 0; q < (over ? n_obj : nl); ++q) {
        const MeshObject& m = obj[over ? (all ? q : s_obj[q]) : s_cell[warp][q]];
        const bool box = pt && !(px < m.lo[0] || px > m.hi[0] || py < m.lo[1] || py > m.hi[1] || pz < m.lo[2] || pz > m.hi[2]);
        int cross = 0;
        if (exact) {
          if (box && holds(m, ci, cj, ck))
            for (int f = 0; f < m.count; ++f) {
              if (TABLES) {
                cross += te[m.entry + f].adet > 0.0 && ray_crosses(px, py, pz, te[m.entry + f]);
              } else {
                MeshTri o;
                mesh_tri(tri + 9 * ((size_t)m.first + f), o);
                cross += o.adet > 0.0 && ray_crosses(px, py, pz, o);
              }
            }
        } else {
          const int end = s_end[warp][q];
          cross = (int)s_odd[warp][q];
          const float lx = (float)((px - m.lo[0]) * m.scale), ly = (float)((py - m.lo[1]) * m.scale), lz = (float)((pz - m.lo[2]) * m.scale);
          for (; at < end; ++at) {
            const int f = s_open[warp][at];
            const int b3 = box ? ray_bound(lx, ly, lz, 0.f, tf[f]) : -1;
            if (b3 == 0) cross += ray_crosses(px, py, pz, te[f]);
            else cross += b3 == 1;
          }
        }
        if (box && (cross & 1)) val = fmin(val, m.phi_in);
      }
      const unsigned int pts = __ballot_sync(0xffffffffu, pt), ones = __ballot_sync(0xffffffffu, pt && val == 1.0);
      const unsigned int zeros = __ballot_sync(0xffffffffu, pt && val == 0.0);
      if (whole && (ones | zeros) == pts) {
        acc += (double)__popc(ones);
      } else {                                       // in sample order
        whole = false;
        s_val[warp][lane] = val;
        __syncwarp();
        for (int l = 0; l < 32 && base + l < npts; ++l) acc = __dadd_rn(acc, s_val[warp][l]);
        __syncwarp();
      }
    }
    if (lane == src) out = (T)__ddiv_rn(acc, (double)npts);
    __syncwarp();
  }
  if (in) phi[(size_t)i + (size_t)P * ((size_t)j + (size_t)ny * k)] = out;
}

}  // namespace uf
