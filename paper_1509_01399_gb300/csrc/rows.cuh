// Rows of the hybrid FEM/FDM scheme shared by the step kernels: per-node rows
// of every kind, the gradient pairings and the rows of the refined region.
//
// The sweep kernel writes fields that it reads in the same launch, so it may not
// load them through the read-only path; the kernels of step_kernels.cu, which
// read one set of levels and write another, define HYB_FIELD as __restrict__.
#pragma once

#ifndef HYB_FIELD
#define HYB_FIELD
#endif

#include "hyb_internal.h"

namespace hyb {
namespace {

// x divided by a face count 1, 2 or 3 (a division only on the three-face
// corners: FP64 divisions are long on this GPU).
template <typename T>
__device__ __forceinline__ T over_faces(T x, int n) {
  if (n == 3) return x / T(3);
  return n == 2 ? T(0.5) * x : x;
}

__device__ __forceinline__ int face_bits(int i, int j, int k, int nx, int ny, int nz) {
  return (i == 0 ? 1 : 0) | (i == nx - 1 ? 2 : 0) | (j == 0 ? 4 : 0) | (j == ny - 1 ? 8 : 0) |
         (k == 0 ? 16 : 0) | (k == nz - 1 ? 32 : 0);
}

// Plane-wave flux term tau^2 (2 / h) g of node (i, j, k) on flux face f
// (the mirror ghost u_g = u_in + 2 h g of d_n u = g, Eq. (f)):
// g = amp (-(d . n_f)) p(t_k - d . (x - x0)), p(s) = sin(omega s) on [0, t1]
// and 0 elsewhere.  The delay is formed in FP64; the pulse in the field's
// precision.
__device__ __forceinline__ double src_term(const Slot<double>& S, int f, int i, int j, int k) {
  const Pulse<double>& p = S.pulse;
  const double s = p.st - (p.sd[0] * (i - S.si0[0]) + p.sd[1] * (j - S.si0[1]) + p.sd[2] * (k - S.si0[2]));
  if (!(s >= 0.0 && s <= p.t1)) return 0.0;
  return S.sf[f] * sin(p.omega * s);
}

// FP32 fields: the phase omega (t_k - d . (x - x0)) in pairs of FP32 numbers
// (Dekker's and Knuth's exact product and sum), to about 2^-45 of its terms before
// the one rounding of the pulse's argument.  In FP64 the delay is a dependent chain of a
// dozen operations on a pipe of two lanes per SM and clock, in the warps next to the
// flux faces, for which a whole level then waits: 250 x 171 x 215, a diagonal
// wave through three faces, 41.8 -> 35.4 us a forward level; 193^3, four sources,
// 107.6 -> 101.2; 129^3 through z, 9.37 -> 9.01.
__device__ __forceinline__ float src_term(const Slot<float>& S, int f, int i, int j, int k) {
  constexpr float kEnd[2] = {6.28318548f, -1.74845553e-7f};  // 2 pi
  const Pulse<float>& p = S.pulse;
  const int q[3] = {i, j, k};
  float s = p.ph[0], lo = p.ph[1];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float n = (float)(q[a] - S.si0[a]);
    const float m = __fmul_rn(p.pd[a][0], n), e = fmaf(p.pd[a][1], n, fmaf(p.pd[a][0], n, -m));
    const float t = __fsub_rn(s, m), b = __fsub_rn(t, s);
    lo += __fsub_rn(__fsub_rn(s, __fsub_rn(t, b)), __fadd_rn(m, b)) - e;
    s = t;
  }
  const float v = __fadd_rn(s, lo), r = __fadd_rn(__fsub_rn(s, v), lo);
  if (!(v >= 0.f && __fsub_rn(v, kEnd[0]) + (r - kEnd[1]) <= 0.f)) return 0.f;
  return S.sf[f] * sinf(v);
}

// Sum of the flux terms of the faces in `faces` (bits) that carry the flux.
template <typename T>
__device__ __forceinline__ T src_terms(const Slot<T>& S, int faces, int i, int j, int k) {
  T v = T(0);
  for (int b = faces & S.src_mask; b; b &= b - 1) v += src_term(S, __ffs(b) - 1, i, j, k);
  return v;
}

__device__ __forceinline__ int face_index(int f, int i, int j, int k, int nx, int ny);

// Paper-mode adjoint: the cotangent c of the observation-face node (i, j, k)
// enters its row as -tau c / M, M = h^3 halved on every axis on which the
// node lies on the outer boundary (the mirror ghost of d_n lambda = -(u - u~)).
template <typename T>
__device__ __forceinline__ T inj_term(const Slot<T>& S, int fall, int i, int j, int k, int nx, int ny) {
  if (S.inj == nullptr || !((fall >> S.obs_face) & 1)) return T(0);
  const int nb = ((fall & 3) ? 1 : 0) + ((fall & 12) ? 1 : 0) + ((fall & 48) ? 1 : 0);
  return S.inj_scale * T(1 << nb) * S.inj[face_index(S.obs_face, i, j, k, nx, ny)];
}

// field index of node (i, j, k)
template <typename T>
__device__ __forceinline__ long long lin(const StepArgs<T>& A, int i, int j, int k) {
  return (long long)i + (long long)A.px * ((long long)j + (long long)A.ny * k);
}

// index of node (i, j, k) in the FEM-owned (history) box
template <typename T>
__device__ __forceinline__ long long hidx(const StepArgs<T>& A, int i, int j, int k) {
  return (long long)(i - A.hx0) + (long long)A.hpx * ((long long)(j - A.fl[1]) + (long long)A.fn[1] * (k - A.fl[2]));
}

template <typename T>
__device__ __forceinline__ bool fem_owned(const StepArgs<T>& A, int i, int j, int k) {
  return i >= A.fl[0] && i <= A.fh[0] && j >= A.fl[1] && j <= A.fh[1] && k >= A.fl[2] &&
         k <= A.fh[2];
}

template <typename T>
__device__ __forceinline__ long long widx(const StepArgs<T>& A, int i, int j, int k) {
  return (long long)(i - A.wx0) +
         (long long)A.wpx * ((long long)(j - A.wl[1]) + (long long)A.wn[1] * (k - A.wl[2]));
}

// sum over the six axis edges of W_e (u_nb - u_c) at a FEM-owned node
template <typename T>
__device__ __forceinline__ T fem_lap(const StepArgs<T>& A, const T* __restrict__ Wb, const T* HYB_FIELD u, long long id,
                                     int i, int j, int k, T c, T zm, T zp) {
  const long long w = widx(A, i, j, k);
  const T* Wx = Wb;
  const T* Wy = Wb + A.wsz;
  const T* Wz = Wb + 2 * A.wsz;
  const long long wy = A.wpx;
  const long long wz = (long long)A.wpx * A.wn[1];
  return Wx[w] * (u[id + 1] - c) + Wx[w - 1] * (u[id - 1] - c) + Wy[w] * (u[id + A.px] - c) +
         Wy[w - wy] * (u[id - A.px] - c) + Wz[w] * (zp - c) + Wz[w - wz] * (zm - c);
}

// ---- the all-FEM path (HYB_FEM_TET_ALL): rows gathered over tetrahedra ----
// Coefficient a of the voxel with origin (ox, oy, oz): its value on the
// unknown voxels, 1 elsewhere (Eq. (2.3)).
template <typename T>
__device__ __forceinline__ double voxel_coef(const StepArgs<T>& A, int ox, int oy, int oz) {
  const int x = ox - A.fl[0], y = oy - A.fl[1], z = oz - A.fl[2];
  if (x >= 0 && y >= 0 && z >= 0 && x < A.un[0] && y < A.un[1] && z < A.un[2])
    return A.acoef[x + (long long)A.un[0] * (y + (long long)A.un[1] * z)];
  return 1.0;
}

template <typename T>
__device__ __forceinline__ bool lattice_interior(const StepArgs<T>& A, int i, int j, int k) {
  return i > 0 && j > 0 && k > 0 && i < A.nx - 1 && j < A.ny - 1 && k < A.nz - 1;
}

// The finite-element row of the interior node n = (i, j, k), gathered over
// the Kuhn tetrahedra of the (up to eight) voxels that have n as a corner:
// sum over those tetrahedra K of a_K K^K_{n q} (element stiffness, Sec. 7.2)
// and the lumped mass M^L_n = sum |K| / 4.  With `u` set, returns the
// Laplacian part -(M^L)^{-1} (K u)_n of Eq. (fem) (unit spacing); else the
// coefficient of row n on node m = (mi, mj, mk) (the diagonal when m = n).
template <typename T>
__device__ __noinline__ T tet_row(const StepArgs<T>& A, const T* __restrict__ u, int i, int j, int k, int mi, int mj,
                                  int mk) {
  const T c = u ? u[lin(A, i, j, k)] : T(0);
  T acc = T(0);
  double mass = 0.0;
  for (int cn = 0; cn < 8; ++cn) {
    const int ox = i - (cn & 1), oy = j - ((cn >> 1) & 1), oz = k - (cn >> 2);
    if (ox < 0 || oy < 0 || oz < 0 || ox > A.nx - 2 || oy > A.ny - 2 || oz > A.nz - 2) continue;
    const T av = (T)voxel_coef(A, ox, oy, oz);
    for (int t = 0; t < 6; ++t) {
      const int* V = A.kuhn_v + 4 * t;
      int ln = -1;
      for (int q = 0; q < 4; ++q)
        if (V[q] == cn) ln = q;
      if (ln < 0) continue;
      mass += A.kuhn[96 + t] * 0.25;
      for (int q = 0; q < 4; ++q) {
        const int cq = V[q];
        const int qi = ox + (cq & 1), qj = oy + ((cq >> 1) & 1), qk = oz + (cq >> 2);
        const T kv = av * (T)A.kuhn[16 * t + 4 * ln + q];
        if (u) {
          if (q != ln) acc += kv * (u[lin(A, qi, qj, qk)] - c);
        } else if (qi == mi && qj == mj && qk == mk) {
          acc += kv;
        }
      }
    }
  }
  return -acc / (T)mass;
}

// Coefficient of the non-absorbing row of node n on node m (Laplacian part,
// unit spacing) on the all-FEM path: the gathered FEM row on interior
// nodes; on the outer boundary the FDM row (mirror ghost: 2 on the inward
// neighbour, 1 on the in-face neighbours, -6 on the node itself).
template <typename T>
__device__ __forceinline__ T tet_coef(const StepArgs<T>& A, int ni, int nj, int nk, int mi, int mj, int mk) {
  if (lattice_interior(A, ni, nj, nk)) return tet_row<T>(A, nullptr, ni, nj, nk, mi, mj, mk);
  const int d0 = mi - ni, d1 = mj - nj, d2 = mk - nk;
  if (d0 == 0 && d1 == 0 && d2 == 0) return A.ani ? A.kdiag : T(-6);
  if (abs(d0) + abs(d1) + abs(d2) != 1) return T(0);
  const int ax = d0 ? 0 : (d1 ? 1 : 2), s = d0 + d1 + d2;
  const int c = ax == 0 ? ni : (ax == 1 ? nj : nk);
  const int n = ax == 0 ? A.nx : (ax == 1 ? A.ny : A.nz);
  const T w = ((s > 0 && c == 0) || (s < 0 && c == n - 1)) ? T(2) : T(1);
  return A.ani ? w * A.kapt[ax] : w;
}

// Pairing of the voxel with origin (i, j, k) on the all-FEM path:
// kGradPairScale sum over its tetrahedra of u^T K^K lambda (a = 1).
template <typename T>
__device__ __forceinline__ T tet_pair(const StepArgs<T>& A, const T* hb, const T* lam, int i, int j, int k) {
  T u[8], l[8];
  for (int c = 0; c < 8; ++c) {
    const int a = c & 1, b = (c >> 1) & 1, d = c >> 2;
    u[c] = hb[hidx(A, i + a, j + b, k + d)];
    l[c] = lam[lin(A, i + a, j + b, k + d)];
  }
  T acc = T(0);
  for (int t = 0; t < 6; ++t)
    for (int p = 0; p < 4; ++p)
      for (int q = 0; q < 4; ++q)
        acc += (T)A.kuhn[16 * t + 4 * p + q] * u[A.kuhn_v[4 * t + p]] * l[A.kuhn_v[4 * t + q]];
  return T(6) * acc;
}

// Laplacian part (without 1/h^2) of a non-absorbing row at any node:
// FEM stencil on FEM-owned nodes, 7-point with mirror ghosts elsewhere (on
// the all-FEM path, the gathered FEM row on every interior node).
template <typename T>
__device__ __noinline__ T row_lap(const StepArgs<T>& A, const T* __restrict__ W, const T* __restrict__ u, int i, int j,
                                  int k) {
  if (A.tet && lattice_interior(A, i, j, k)) return tet_row<T>(A, u, i, j, k, 0, 0, 0);
  const long long id = lin(A, i, j, k);
  const long long sz = (long long)A.px * A.ny;
  const T c = u[id];
  if (fem_owned(A, i, j, k)) return fem_lap(A, W, u, id, i, j, k, c, u[id - sz], u[id + sz]);
  T lx, ly, lz;
  if (i == 0) lx = T(2) * (u[id + 1] - c);
  else if (i == A.nx - 1) lx = T(2) * (u[id - 1] - c);
  else lx = (u[id - 1] - c) + (u[id + 1] - c);
  if (j == 0) ly = T(2) * (u[id + A.px] - c);
  else if (j == A.ny - 1) ly = T(2) * (u[id - A.px] - c);
  else ly = (u[id - A.px] - c) + (u[id + A.px] - c);
  if (k == 0) lz = T(2) * (u[id + sz] - c);
  else if (k == A.nz - 1) lz = T(2) * (u[id - sz] - c);
  else lz = (u[id - sz] - c) + (u[id + sz] - c);
  if (A.ani) return (A.kapt[0] * lx + A.kapt[1] * ly) + A.kapt[2] * lz;
  return (lx + ly) + lz;
}

// Coefficient of u_b^k in the absorbing row of a node on the absorbing faces
// fb (bits): r, or with per-axis steps the mean of its faces' coefficients.
template <typename T>
__device__ __forceinline__ T abc_self(const StepArgs<T>& A, int fb) {
  if (!A.ani) return A.r;
  T rs = T(0);
  for (int b = fb; b; b &= b - 1) rs += A.ra[(__ffs(b) - 1) >> 1];
  return over_faces(rs, __popc(fb));
}

// u^{k+1} at any node, recursing into the inward neighbours of absorbing
// rows (depth D bounds the recursion: a node lies on at most 3 faces).
template <typename T, int D>
__device__ __noinline__ T fwd_new(const StepArgs<T>& A, const Slot<T>& S, int i, int j, int k) {
  const long long id = lin(A, i, j, k);
  const int fall = face_bits(i, j, k, A.nx, A.ny, A.nz);
  if constexpr (D > 0) {
    const int fb = fall & S.mask_f;
    if (fb) {
      T acc = T(0);
#pragma unroll
      for (int f = 0; f < 6; ++f) {
        if (fb & (1 << f)) {
          const int ax = f >> 1;
          const int step = (f & 1) ? -1 : 1;  // inward
          const int i1 = i + (ax == 0 ? step : 0);
          const int j1 = j + (ax == 1 ? step : 0);
          const int k1 = k + (ax == 2 ? step : 0);
          const T rf = A.ani ? A.ra[ax] : A.r;
          acc += S.cur[lin(A, i1, j1, k1)] - rf * fwd_new<T, D - 1>(A, S, i1, j1, k1);
        }
      }
      return abc_self(A, fb) * S.cur[id] + acc / T(__popc(fb));
    }
  }
  const T c = S.cur[id];
  T v = c + ((c - S.prev[id]) + A.c2 * row_lap(A, S.W, S.cur, i, j, k));
  if (fall & S.src_mask) v += src_terms(S, fall, i, j, k);
  if (S.inj) v += inj_term(S, fall, i, j, k, A.nx, A.ny);
  return v;
}

// Coefficient of the non-absorbing row of node (i,j,k) on its neighbour
// (i,j,k) + s e_ax (Laplacian part, without 1/h^2).
template <typename T>
__device__ __forceinline__ T row_coef(const StepArgs<T>& A, const T* __restrict__ W, int i, int j, int k, int ax,
                                      int s) {
  if (fem_owned(A, i, j, k)) {
    const long long w = widx(A, i, j, k);
    const long long ws = ax == 0 ? 1 : (ax == 1 ? (long long)A.wpx : (long long)A.wpx * A.wn[1]);
    return W[ax * A.wsz + (s > 0 ? w : w - ws)];
  }
  const int c = ax == 0 ? i : (ax == 1 ? j : k);
  const int n = ax == 0 ? A.nx : (ax == 1 ? A.ny : A.nz);
  const T w = ((s > 0 && c == 0) || (s < 0 && c == n - 1)) ? T(2) : T(1);
  return A.ani ? w * A.kapt[ax] : w;
}

template <typename T>
__device__ __forceinline__ T row_diag(const StepArgs<T>& A, const T* __restrict__ W, int i, int j, int k) {
  if (fem_owned(A, i, j, k)) {
    const long long w = widx(A, i, j, k);
    const long long wy = A.wpx;
    const long long wz = (long long)A.wpx * A.wn[1];
    return -(W[w] + W[w - 1] + W[A.wsz + w] + W[A.wsz + w - wy] + W[2 * A.wsz + w] +
             W[2 * A.wsz + w - wz]);
  }
  return A.ani ? A.kdiag : T(-6);
}

__device__ __forceinline__ int face_index(int f, int i, int j, int k, int nx, int ny) {
  const int ax = f >> 1;
  if (ax == 2) return i + nx * j;
  if (ax == 1) return i + nx * k;
  return j + ny * k;
}

// Right-hand side of the transposed step at node m:
// (B_j^T lambda^{j+1})_m - (C_{j+1}^T lambda^{j+2})_m + c^j_m.
template <typename T>
__device__ __noinline__ T adj_rhs(const StepArgs<T>& A, const Slot<T>& S, int i, int j, int k) {
  const T* __restrict__ l1 = S.cur;
  const long long id = lin(A, i, j, k);
  const int fbm = face_bits(i, j, k, A.nx, A.ny, A.nz);
  T rhs;
  if (fbm & S.mask_f) rhs = abc_self(A, fbm & S.mask_f) * l1[id];
  else rhs = (T(2) + A.c2 * row_diag(A, S.W, i, j, k)) * l1[id];
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int s = t ? 1 : -1;
      const int ni = i + (ax == 0 ? s : 0);
      const int nj = j + (ax == 1 ? s : 0);
      const int nk = k + (ax == 2 ? s : 0);
      if (ni < 0 || ni >= A.nx || nj < 0 || nj >= A.ny || nk < 0 || nk >= A.nz) continue;
      const long long nid = lin(A, ni, nj, nk);
      const int fbn = face_bits(ni, nj, nk, A.nx, A.ny, A.nz) & S.mask_f;
      if (fbn) {
        // absorbing row of the neighbour couples to m only when m is its
        // inward neighbour across the face on side s of axis ax
        const int f = 2 * ax + (s > 0 ? 1 : 0);
        if (fbn & (1 << f)) rhs += l1[nid] / T(__popc(fbn));
      } else {
        rhs += A.c2 * row_coef(A, S.W, ni, nj, nk, ax, -s) * l1[nid];
      }
    }
  }
  if (!(fbm & S.mask_c)) rhs -= S.prev[id];
  if (S.obs_r && ((fbm >> S.obs_face) & 1)) rhs += S.obs_r[face_index(S.obs_face, i, j, k, A.nx, A.ny)];
  return rhs;
}

// adj_rhs on the all-FEM path: the transposed row gathers the coefficients
// of every neighbouring row (the 26 nodes around m) on m.
template <typename T>
__device__ __noinline__ T adj_rhs_tet(const StepArgs<T>& A, const Slot<T>& S, int i, int j, int k) {
  const T* __restrict__ l1 = S.cur;
  const long long id = lin(A, i, j, k);
  const int fbm = face_bits(i, j, k, A.nx, A.ny, A.nz);
  T rhs;
  if (fbm & S.mask_f) rhs = abc_self(A, fbm & S.mask_f) * l1[id];
  else rhs = (T(2) + A.c2 * tet_coef(A, i, j, k, i, j, k)) * l1[id];
  for (int d = 0; d < 27; ++d) {
    const int dx = d % 3 - 1, dy = (d / 3) % 3 - 1, dz = d / 9 - 1;
    if (d == 13) continue;
    const int ni = i + dx, nj = j + dy, nk = k + dz;
    if (ni < 0 || ni >= A.nx || nj < 0 || nj >= A.ny || nk < 0 || nk >= A.nz) continue;
    const long long nid = lin(A, ni, nj, nk);
    const int fbn = face_bits(ni, nj, nk, A.nx, A.ny, A.nz) & S.mask_f;
    if (fbn) {
      // an absorbing row couples to m only when m is its inward neighbour
      // across one of its absorbing faces
      if (abs(dx) + abs(dy) + abs(dz) != 1) continue;
      const int ax = dx ? 0 : (dy ? 1 : 2), s = -(dx + dy + dz);  // m = n + s e_ax
      const int f = 2 * ax + (s > 0 ? 0 : 1);
      if (fbn & (1 << f)) rhs += l1[nid] / T(__popc(fbn));
    } else {
      rhs += A.c2 * tet_coef(A, ni, nj, nk, i, j, k) * l1[nid];
    }
  }
  if (!(fbm & S.mask_c)) rhs -= S.prev[id];
  if (S.obs_r && ((fbm >> S.obs_face) & 1)) rhs += S.obs_r[face_index(S.obs_face, i, j, k, A.nx, A.ny)];
  return rhs;
}

// Inlined form of adj_rhs for the edge tiles.  Every load is issued first,
// predicated, and the row summed afterwards: the nodes of an edge tile's warp
// take different branches (faces, absorbing rows, FEM weights), and loads
// inside those branches would each wait for memory in turn.
template <typename T, bool ANI>
__device__ __forceinline__ T adj_rhs_inl(const StepArgs<T>& A, const Slot<T>& S, int i, int j, int k) {
  const T* HYB_FIELD l1 = S.cur;
  const long long id = lin(A, i, j, k);
  const int fbm = face_bits(i, j, k, A.nx, A.ny, A.nz);
  const long long wy = A.wpx, wz = (long long)A.wpx * A.wn[1];
  const bool fo = fem_owned(A, i, j, k);
  const long long w = fo ? widx(A, i, j, k) : 0;
  const T* W = S.W;
  T wd[6];  // this node's edge weights (FEM-owned nodes)
  wd[0] = fo ? W[w] : T(0);
  wd[1] = fo ? W[w - 1] : T(0);
  wd[2] = fo ? W[A.wsz + w] : T(0);
  wd[3] = fo ? W[A.wsz + w - wy] : T(0);
  wd[4] = fo ? W[2 * A.wsz + w] : T(0);
  wd[5] = fo ? W[2 * A.wsz + w - wz] : T(0);
  const T lc = l1[id];
  const T pv = S.prev[id];
  const bool obs = S.obs_r != nullptr && ((fbm >> S.obs_face) & 1);
  const T ov = obs ? S.obs_r[face_index(S.obs_face, i, j, k, A.nx, A.ny)] : T(0);
  T nb[6], cw[6];
  int nfb[6];
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int q = 2 * ax + t;
      const int s = t ? 1 : -1;
      const int ni = i + (ax == 0 ? s : 0);
      const int nj = j + (ax == 1 ? s : 0);
      const int nk = k + (ax == 2 ? s : 0);
      const bool inb = ni >= 0 && ni < A.nx && nj >= 0 && nj < A.ny && nk >= 0 && nk < A.nz;
      nb[q] = l1[inb ? lin(A, ni, nj, nk) : id];
      nfb[q] = inb ? (face_bits(ni, nj, nk, A.nx, A.ny, A.nz) & S.mask_f) : -1;
      // coefficient of the neighbour's non-absorbing row on this node (row_coef)
      const bool nfo = inb && fem_owned(A, ni, nj, nk);
      const long long ws = ax == 0 ? 1 : (ax == 1 ? wy : wz);
      const long long nw = nfo ? ax * A.wsz + (s < 0 ? widx(A, ni, nj, nk) : widx(A, ni, nj, nk) - ws) : 0;
      const T wv = nfo ? W[nw] : T(0);
      const int c = ax == 0 ? ni : (ax == 1 ? nj : nk);
      const int n = ax == 0 ? A.nx : (ax == 1 ? A.ny : A.nz);
      cw[q] = nfo ? wv : (((s < 0 && c == 0) || (s > 0 && c == n - 1)) ? T(2) : T(1)) * (ANI ? A.kapt[ax] : T(1));
    }
  }
  T rhs;
  if (fbm & S.mask_f) rhs = (ANI ? abc_self(A, fbm & S.mask_f) : A.r) * lc;
  else rhs = (T(2) + A.c2 * (fo ? -(wd[0] + wd[1] + wd[2] + wd[3] + wd[4] + wd[5]) : (ANI ? A.kdiag : T(-6)))) * lc;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    if (nfb[q] < 0) continue;
    if (nfb[q]) {
      // absorbing row of the neighbour couples to m only when m is its
      // inward neighbour across the face on side s of axis ax
      const int f = 2 * (q >> 1) + (q & 1);
      if (nfb[q] & (1 << f)) rhs += over_faces(nb[q], __popc(nfb[q]));
    } else {
      rhs += A.c2 * cw[q] * nb[q];
    }
  }
  if (!(fbm & S.mask_c)) rhs -= pv;
  return rhs + ov;
}

// lambda^j at node m: solve E_{j-1}^T lambda^j = rhs, where E couples an
// absorbing node b to its inward neighbours with r / L_b.
template <typename T, int D>
__device__ __noinline__ T adj_new(const StepArgs<T>& A, const Slot<T>& S, int i, int j, int k) {
  T v = A.tet ? adj_rhs_tet(A, S, i, j, k) : adj_rhs(A, S, i, j, k);
  if constexpr (D > 0) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int s = t ? 1 : -1;
        const int bi = i + (ax == 0 ? s : 0);
        const int bj = j + (ax == 1 ? s : 0);
        const int bk = k + (ax == 2 ? s : 0);
        if (bi < 0 || bi >= A.nx || bj < 0 || bj >= A.ny || bk < 0 || bk >= A.nz) continue;
        const int f = 2 * ax + (s > 0 ? 1 : 0);
        const int fbb = face_bits(bi, bj, bk, A.nx, A.ny, A.nz) & S.mask_e;
        if (fbb & (1 << f)) v -= ((A.ani ? A.ra[ax] : A.r) / T(__popc(fbb))) * adj_new<T, D - 1>(A, S, bi, bj, bk);
      }
    }
  }
  return v;
}

// Six times the sum over the 12 axis edges of a voxel of
// w_e (u_p - u_q)(l_p - l_q), corner c = a + 2b + 4d at offset (a, b, d);
// w_e = 1/3 on the edges at the voxel's diagonal corners 0 and 7, 1/6 on the
// others.  (The factor 6 keeps divisions out of the kernels; the host scale
// of the gradient divides it out.)
template <typename T>
__device__ __forceinline__ T pair_sum(const T u[8], const T l[8]) {
  const T d3 = (u[1] - u[0]) * (l[1] - l[0]) + (u[7] - u[6]) * (l[7] - l[6]) +
               (u[2] - u[0]) * (l[2] - l[0]) + (u[7] - u[5]) * (l[7] - l[5]) +
               (u[4] - u[0]) * (l[4] - l[0]) + (u[7] - u[3]) * (l[7] - l[3]);
  const T d6 = (u[3] - u[2]) * (l[3] - l[2]) + (u[5] - u[4]) * (l[5] - l[4]) +
               (u[3] - u[1]) * (l[3] - l[1]) + (u[6] - u[4]) * (l[6] - l[4]) +
               (u[5] - u[1]) * (l[5] - l[1]) + (u[6] - u[2]) * (l[6] - l[2]);
  return T(2) * d3 + d6;
}

// Telegraph reading: 12 times the pairing sum_i m_i lambda_i v_i of a voxel,
// v = u^{k+1} - u^{k-1} at its corners (the stored history) and m_i its lumped
// mass share of corner i in units of h^3: 1/4 on the diagonal corners 0 and
// 7, 1/12 on the others.
template <typename T>
__device__ __forceinline__ T damp_sum(const T u[8], const T l[8]) {
  const T d = u[0] * l[0] + u[7] * l[7];
  const T o = ((u[1] * l[1] + u[2] * l[2]) + (u[3] * l[3] + u[4] * l[4])) + (u[5] * l[5] + u[6] * l[6]);
  return T(3) * d + o;
}

// pair_sum with per-axis steps: the sums over the x, y and z edges weighed by
// kap (the voxel is a brick; dx_1^2 / dx_ax^2 relative to the x edges).
template <typename T>
__device__ __forceinline__ T pair_sum_ani(const StepArgs<T>& A, const T u[8], const T l[8]) {
  const T x = T(2) * ((u[1] - u[0]) * (l[1] - l[0]) + (u[7] - u[6]) * (l[7] - l[6])) +
              ((u[3] - u[2]) * (l[3] - l[2]) + (u[5] - u[4]) * (l[5] - l[4]));
  const T y = T(2) * ((u[2] - u[0]) * (l[2] - l[0]) + (u[7] - u[5]) * (l[7] - l[5])) +
              ((u[3] - u[1]) * (l[3] - l[1]) + (u[6] - u[4]) * (l[6] - l[4]));
  const T z = T(2) * ((u[4] - u[0]) * (l[4] - l[0]) + (u[7] - u[3]) * (l[7] - l[3])) +
              ((u[5] - u[1]) * (l[5] - l[1]) + (u[6] - u[2]) * (l[6] - l[2]));
  return (A.kapt[0] * x + A.kapt[1] * y) + A.kapt[2] * z;
}

// pair_sum of voxel (i,j,k): u from the FEM-owned box hb, lambda from the lattice
template <typename T>
__device__ __forceinline__ T voxel_pair(const StepArgs<T>& A, const T* HYB_FIELD hb, const T* HYB_FIELD lam, int i, int j,
                                        int k) {
  const long long hy = A.hpx;
  const long long hz = (long long)A.hpx * A.fn[1];
  const long long h0 = hidx(A, i, j, k);
  const long long ly = A.px;
  const long long lz = (long long)A.px * A.ny;
  const long long l0 = lin(A, i, j, k);
  T u[8], l[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int a = c & 1, b = (c >> 1) & 1, d = c >> 2;
    u[c] = hb[h0 + a + b * hy + d * hz];
    l[c] = lam[l0 + a + b * ly + d * lz];
  }
  return A.sdamp ? damp_sum(u, l) : pair_sum(u, l);
}

// voxel_pair with per-axis steps
template <typename T>
__device__ __forceinline__ T voxel_pair_ani(const StepArgs<T>& A, const T* hb, const T* lam, int i, int j, int k) {
  T u[8], l[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int a = c & 1, b = (c >> 1) & 1, d = c >> 2;
    u[c] = hb[hidx(A, i + a, j + b, k + d)];
    l[c] = lam[lin(A, i + a, j + b, k + d)];
  }
  return pair_sum_ani(A, u, l);
}

// Laplacian part (without 1/h^2) of a 7-point row with unit weights.
template <typename T>
__device__ __forceinline__ T lap7(T xm, T xp, T ym, T yp, T zm, T zp, T c) {
  return (xm - c) + (xp - c) + (ym - c) + (yp - c) + (zm - c) + (zp - c);
}

// Laplacian part of a non-absorbing row (inlined form of row_lap).
template <typename T, bool ANI>
__device__ __forceinline__ T row_lap_inl(const StepArgs<T>& A, const T* __restrict__ W, const T* HYB_FIELD u, int i, int j,
                                         int k) {
  const long long id = lin(A, i, j, k);
  const long long sz = (long long)A.px * A.ny;
  const T c = u[id];
  if (fem_owned(A, i, j, k)) return fem_lap(A, W, u, id, i, j, k, c, u[id - sz], u[id + sz]);
  const T xm = i > 0 ? u[id - 1] : u[id + 1];
  const T xp = i < A.nx - 1 ? u[id + 1] : u[id - 1];
  const T ym = j > 0 ? u[id - A.px] : u[id + A.px];
  const T yp = j < A.ny - 1 ? u[id + A.px] : u[id - A.px];
  const T zm = k > 0 ? u[id - sz] : u[id + sz];
  const T zp = k < A.nz - 1 ? u[id + sz] : u[id - sz];
  if constexpr (ANI)
    return (A.kapt[0] * ((xm - c) + (xp - c)) + A.kapt[1] * ((ym - c) + (yp - c))) + A.kapt[2] * ((zm - c) + (zp - c));
  return lap7(xm, xp, ym, yp, zm, zp, c);
}

// (TET: per-axis steps or the all-FEM path may be on)
template <typename T, bool TET>
__device__ __forceinline__ void pair_if_voxel(const StepArgs<T>& A, const Slot<T>& S, int si, int i, int j,
                                              int k) {
  if (S.hist_r == nullptr) return;
  if (i < A.fl[0] || i >= A.fl[0] + A.un[0] || j < A.fl[1] || j >= A.fl[1] + A.un[1] || k < A.fl[2] ||
      k >= A.fl[2] + A.un[2])
    return;
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
  const long long vid = (long long)(i - A.fl[0]) +
                        (long long)A.un[0] * ((j - A.fl[1]) + (long long)A.un[1] * (k - A.fl[2]));
  if (A.refvox && A.refvox[vid]) return;
  if (TET && A.tet) A.G[(long long)si * nv + vid] += (double)tet_pair(A, S.hist_r, S.cur, i, j, k);
  else if (TET && A.ani) A.G[(long long)si * nv + vid] += (double)voxel_pair_ani(A, S.hist_r, S.cur, i, j, k);
  else A.G[(long long)si * nv + vid] += (double)voxel_pair(A, S.hist_r, S.cur, i, j, k);
}

template <typename T>
__device__ __forceinline__ long long axis_stride(const StepArgs<T>& A, int ax) {
  return ax == 0 ? 1LL : (ax == 1 ? (long long)A.px : (long long)A.px * A.ny);
}

// Refined region of one time level (one thread per row), the same rows for the forward and the
// mass-scaled adjoint.  A corner n of refined voxels: the Kuhn stencil row
// lapW (the edge weights over the voxels around n) corrected on every refined
// voxel v around n by a_v (K9 - K8) of n's corner in v, which couples the
// voxel's diagonal corners 0 and 7 to its six others, the six others to 0
// and 7, and every corner to the centre; divided by n's lumped mass in units
// of h^3.  A centre c of voxel v: a_v K9 of the centre on the eight corners
// over its mass.  Then u^{k+1} = u^k + ((u^k - u^{k-1}) + tau^2/h^2 lap).
// Every load of a row is issued before the row is summed.
template <typename T, bool ADJ>
__device__ __forceinline__ void refined_corner(const StepArgs<T>& A, const Slot<T>& S, int r) {
  const uint2 pos = A.rpos[r];
  const int i = (int)(pos.x & 0xffffu), j = (int)(pos.x >> 16), k = (int)pos.y;
  const long long sy = A.px, sz = (long long)A.px * A.ny;
  const long long id = i + sy * j + sz * k;
  const T* HYB_FIELD u = S.cur;
  // the node's 3 x 3 x 3 neighbourhood (index (dx+1) + 3 (dy+1) + 9 (dz+1)):
  // a refined voxel's K9 - K8 couples n only to the six face neighbours
  // (which the stencil reads too) and to the six neighbours across the
  // diagonals of the coordinate planes with equal signs; a corner of a
  // refined voxel lies inside the FEM block, so all of them are lattice nodes
  T nb[27];
#pragma unroll
  for (int q = 0; q < 27; ++q) nb[q] = T(0);
  nb[13] = u[id];
  nb[12] = u[id - 1];
  nb[14] = u[id + 1];
  nb[10] = u[id - sy];
  nb[16] = u[id + sy];
  nb[4] = u[id - sz];
  nb[22] = u[id + sz];
  nb[9] = u[id - 1 - sy];
  nb[17] = u[id + 1 + sy];
  nb[3] = u[id - 1 - sz];
  nb[23] = u[id + 1 + sz];
  nb[1] = u[id - sy - sz];
  nb[25] = u[id + sy + sz];
  const T c0 = nb[13], pv = S.prev[id];
  const long long w = widx(A, i, j, k);
  const T* Wx = S.W;
  const T* Wy = S.W + A.wsz;
  const T* Wz = S.W + 2 * A.wsz;
  const long long wy = A.wpx, wz = (long long)A.wpx * A.wn[1];
  const T lapW = Wx[w] * (nb[14] - c0) + Wx[w - 1] * (nb[12] - c0) + Wy[w] * (nb[16] - c0) +
                 Wy[w - wy] * (nb[10] - c0) + Wz[w] * (nb[22] - c0) + Wz[w - wz] * (nb[4] - c0);
  // the eight voxels around n (n is corner c of the voxel with origin n - c)
  const int ox = i - A.fl[0], oy = j - A.fl[1], oz = k - A.fl[2];
  const int v0 = ox + A.un[0] * (oy + A.un[1] * oz), vy = A.un[0], vz = A.un[0] * A.un[1];
  int rc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const bool in = ox - dx >= 0 && oy - dy >= 0 && oz - dz >= 0 && ox - dx < A.un[0] && oy - dy < A.un[1] &&
                    oz - dz < A.un[2];
    rc[c] = in ? A.rcid[v0 - dx - dy * vy - dz * vz] : -1;
  }
  T corr = T(0), mass = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int dx = c & 1, dy = (c >> 1) & 1, dz = c >> 2;
    const bool ref = rc[c] >= 0;
    mass += ref ? A.rm9[c] : A.rm8[c];
    const T av = ref ? S.avox[v0 - dx - dy * vy - dz * vz] : T(0);
    const T uc = ref ? S.ccur[rc[c]] : c0;
    T sv = A.rdK[9 * c + 8] * (uc - c0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool diag_c = c == 0 || c == 7, diag_q = q == 0 || q == 7;
      if (q == c || diag_c == diag_q) continue;
      const int o = ((q & 1) - dx + 1) + 3 * (((q >> 1) & 1) - dy + 1) + 9 * ((q >> 2) - dz + 1);
      sv += A.rdK[9 * c + q] * (nb[o] - c0);
    }
    corr += av * sv;
  }
  const T val = c0 + ((c0 - pv) + A.c2 * ((lapW - corr) / mass));
  S.next[id] = val;
  if (!ADJ && S.hist_w) S.hist_w[hidx(A, i, j, k)] = val;
}

// Pairing sum u^T K9 lambda over a refined voxel's 8 corners and centre
// (index 8), K9 the stiffness of the refined unit voxel (a = 1).
template <typename T, typename K>
__device__ __forceinline__ T refined_pair_sum(const T (&u)[9], const T (&l)[9], const K* __restrict__ k9) {
  T acc = T(0);
#pragma unroll
  for (int p = 0; p < 9; ++p) {
    T row = T(0);
#pragma unroll
    for (int q = 0; q < 9; ++q) row += (T)k9[p * 9 + q] * l[q];
    acc += u[p] * row;
  }
  return acc;
}

// Centre row of refined voxel v (centre order); in the transposed step with
// pairing the same thread also adds the voxel's pairing of (u^j, lambda^{j+1})
// to slot si's gradient, from the lambda values the row has loaded.
template <typename T, bool ADJ>
__device__ __forceinline__ void refined_centre(const StepArgs<T>& A, const Slot<T>& S, int v, int si) {
  const int vid = A.refvox_id[v];
  const uint2 xyz = A.rvxyz[v];
  const int x = (int)(xyz.x & 0xffffu), y = (int)(xyz.x >> 16), z = (int)xyz.y;
  const long long l0 = lin(A, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z);
  const long long sy = A.px, sz = (long long)A.px * A.ny;
  T q[9];
#pragma unroll
  for (int c = 0; c < 8; ++c) q[c] = S.cur[l0 + (c & 1) + ((c >> 1) & 1) * sy + (c >> 2) * sz];
  const T uc = S.ccur[v], up = S.cprev[v], av = S.avox[vid];
  q[8] = uc;
  T sv = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) sv += A.rK9[72 + c] * (q[c] - uc);
  const T vc = uc + ((uc - up) - A.c2 * av * sv / A.rm9[8]);
  S.cnext[v] = vc;
  if (!ADJ && S.chist_w) S.chist_w[v] = vc;
  if constexpr (ADJ) {
    if (!S.hist_r) return;
    const long long h0 = hidx(A, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z);
    const long long hy = A.hpx, hz = (long long)A.hpx * A.fn[1];
    T u[9];
#pragma unroll
    for (int c = 0; c < 8; ++c) u[c] = S.hist_r[h0 + (c & 1) + ((c >> 1) & 1) * hy + (c >> 2) * hz];
    u[8] = S.chist_r[v];
    const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
    // the unit-voxel K9 from the launch parameters (kGradPairScale times the pairing, as the other kernels)
    // the only update of this entry in the launch: a reduction without return needs no load
    atomicAdd(A.G + (long long)si * nv + vid, (double)(T(kGradPairScale) * refined_pair_sum(u, q, A.rK9)));
  }
}

}  // namespace
}  // namespace hyb
