// Time-step kernels of the hybrid FEM/FDM scheme.
//
// One time level of every slot (source / problem) is one launch of
// step_kernel: its leading blocks run the edge tiles (nodes within one node
// of two faces), the next ones the interior (all other nodes), one work item
// (slot, 32 x 16 tile, z range) each, and its trailing blocks the rows of
// the refined region.  All
// blocks read levels k and k-1 and write disjoint nodes of level k+1.  An
// interior block's producer warp stages the planes it needs (u^k with a
// one-node halo, u^{k-1}, FEM edge weights, stored history) into shared
// memory with bulk tensor copies, one level ahead on items with FEM-owned
// nodes and six on the others (which stage only u^k and u^{k-1}); its
// eight consumer warps (two tile rows per thread) march the z range reading
// only shared memory, synchronised with the producer by per-level mbarriers
// only.  In tiles with one x face, lanes of the producer warp compute the
// column next to that face.  Consecutive launches overlap through
// programmatic dependent launch.
// Row kinds:
//  * FDM rows, Eq. (fdmschemeforward): u^{k+1} = 2u^k - u^{k-1} + tau^2 Delta_h u^k,
//  * FEM rows on the FEM-owned nodes, Eq. (fem) with lumped mass: on the
//    Kuhn-cut voxels the row is a 7-point stencil whose axis-edge weight is
//    W = sum over the four voxels around the edge of a_c / 3 (edge touching
//    the voxel's diagonal corners) or a_c / 6,
//  * boundary rows: Neumann mirror ghosts, the plane-wave flux of Eq. (f),
//    and the absorbing rows of Eq. (eq:abs2), which use the new value of the
//    inward neighbour: the thread of that neighbour writes the face node, and
//    edge/corner threads recompute the values they need, so no intra-step
//    synchronisation between blocks is needed.
// Both schemes write the same field, so the omega_o / omega_diamond copies
// of Algorithm 1 need no data movement.
//
// The transposed step is the exact transpose of the forward step (the
// discrete form of Eq. (adjoint1)).  Away from the outer boundary the
// mass-weighted operator is symmetric, so the transposed row is the forward
// stencil; next to a face the transposed face row (closed form) and its
// coupling are added, and near edges each node gathers the transposed
// coefficients of its neighbours' rows (mirror factors, absorbing rows) and
// solves the transposed absorbing coupling by recomputing the outer values.
// The same launch accumulates, per unknown voxel and in FP64, the sum over
// the voxel's 12 axis edges of w_e (u_p - u_q)(lambda_p - lambda_q) with
// w_e = 2 or 1 (six times the edge weights 1/3 and 1/6); the host scales it
// by -tau^2 / (6 h^2) (Eq. (gradient1)).
//
// Lattices whose steps differ per axis (ANI) weigh the axis terms by kap and take
// the faces' own absorbing coefficients, by variants of the same kernel without
// refinement (those weights are operands from the argument block and cost no
// registers): 257 x 193 x 321, eight sources, 0.37 / 0.43 ms a level (forward /
// transposed), 0.95 / 2.11 ms by two kernels over the nodes and 0.52 / 0.71 ms by
// the sweep kernel before.
//
// FP64 fields take the sweep kernel (sweep_kernels.cu) instead of step_kernel;
// lattices with fewer than 5 nodes on an axis and the all-FEM path one generic
// kernel over every node.
#define HYB_FIELD __restrict__
#include "async_copy.cuh"
#include "rows.cuh"

namespace hyb {
namespace {

// The "edge set" (lattices with >= 5 nodes per axis): every node whose
// coordinate is near a face (0, 1, n-2 or n-1) on at least two axes.  It is
// cut into tiles of 128 threads: tile 0 is the 4 x 4 x 4 corner block
// (threads 0..63), the other tiles are 8 consecutive positions of one of
// the 12 edge bars (4 x 4 near coordinates x 8).  Within a tile every
// absorbing coupling stays inside the tile.  Returns false for idle threads;
// q[] holds the near index (0..3 -> 0, 1, n-2, n-1) per axis (-1: mid) and
// nf the number of axes on which the node is on a face.
template <typename T>
__device__ __forceinline__ bool edge_tile_node(const StepArgs<T>& A, int blk, int t, int& i, int& j, int& k,
                                               int q[3], int& nf) {
  const int nx = A.nx, ny = A.ny, nz = A.nz;
  auto nr = [](int qq, int n) { return qq < 2 ? qq : n - 4 + qq; };
  int pos = 0, bar = -1;
  if (blk == 0) {
    if (t >= 64) return false;
    q[0] = t & 3;
    q[1] = (t >> 2) & 3;
    q[2] = t >> 4;
  } else {
    blk -= 1;
    const int bz = (nz - 4 + 7) / 8, by = (ny - 4 + 7) / 8;
    const int lo = t & 3, hi = (t >> 2) & 3;
    if (blk < bz) {
      bar = 2;
      pos = blk * 8 + (t >> 4);
      if (pos >= nz - 4) return false;
      q[0] = lo;
      q[1] = hi;
      q[2] = -1;
    } else if (blk < bz + by) {
      bar = 1;
      pos = (blk - bz) * 8 + (t >> 4);
      if (pos >= ny - 4) return false;
      q[0] = lo;
      q[1] = -1;
      q[2] = hi;
    } else {
      bar = 0;
      pos = (blk - bz - by) * 8 + (t >> 4);
      if (pos >= nx - 4) return false;
      q[0] = -1;
      q[1] = lo;
      q[2] = hi;
    }
  }
  i = q[0] < 0 ? 2 + pos : nr(q[0], nx);
  j = q[1] < 0 ? 2 + pos : nr(q[1], ny);
  k = q[2] < 0 ? 2 + pos : nr(q[2], nz);
  nf = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) nf += (q[a] == 0 || q[a] == 3) ? 1 : 0;
  (void)bar;
  return true;
}

// Thread index, inside the same tile, of the node with near index qn on
// axis ax (the other coordinates unchanged).
__device__ __forceinline__ int edge_tile_peer(int t, int blk, const int q[3], int ax, int qn) {
  if (blk == 0) {
    const int sh = 2 * ax;
    return (t & ~(3 << sh)) | (qn << sh);
  }
  // bar tiles: bits 0-1 = first near axis, bits 2-3 = second near axis
  int first = -1;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (q[a] >= 0) {
      first = a;
      break;
    }
  const int sh = (ax == first) ? 0 : 2;
  return (t & ~(3 << sh)) | (qn << sh);
}

// Position of an interior thread.
struct Col {
  int si, i, j;
  int dxs, dys;   // -1 / +1: one node inside the low / high face of x, y; 0: not
  bool xy_fem;    // (i, j) inside the FEM-owned range
  bool xy_uv;     // (i, j) is the x-y origin of an unknown voxel
  bool xy_vox;    // ... and the step pairs
  int rz0, rz1;   // z range of the column's sparse-row nodes (rz0 > rz1: none)
};

// ---- shared-memory pipeline of the interior blocks ----
// A block stages, plane by plane and kPipe<T>::D levels ahead of its z
// march, boxes that its producer warp loads with bulk tensor copies (TMA):
// u^k on the tile and a one-node halo (Box: the box starts on a 16-byte
// boundary, hx columns left of the tile, and is BX x 18), u^{k-1} on the
// same box, and on tiles that meet the FEM block the three edge-weight
// arrays and, for the transposed step, the stored u of the FEM-owned box
// (BX x 17).  Each plane lives in a ring of stages indexed by the plane
// number modulo the ring size.  The copies of a level complete on its "full"
// mbarrier; each of the eight consumer warps (the 32 x 16 tile, two rows per
// thread) waits on it, reads only shared memory and arrives on the level's
// "empty" mbarrier, on which the producer waits before it overwrites the
// level's stages.  The consumer warps thus run up to D levels apart.
// stage of plane k in a ring of N stages (k >= 0)
template <int N>
__device__ __forceinline__ int ring(int k) {
  return (int)((unsigned)k % (unsigned)N);
}

template <typename T>
struct kPipe {
  static constexpr int pow2(int n) { return n <= 1 ? 1 : 2 * pow2((n + 1) / 2); }
  static constexpr int round128(int elems) { return (int)(((elems * (int)sizeof(T) + 127) / 128) * 128 / sizeof(T)); }
  static constexpr int D = 1;             // levels in flight (tiles meeting the FEM block)
  static constexpr int SC = D + 3;        // u^k stages (planes k-1 .. k+1+D)
  static constexpr int SP = pow2(D + 1);  // u^{k-1} stages (k .. k+D)
  static constexpr int SW = D + 2;        // edge-weight stages (k-1 .. k+D)
  static constexpr int SH = D + 2;        // stored-u stages (k .. k+1+D)
  static constexpr int NB = pow2(D + 1);  // level barriers (of each kind)
  static constexpr int CS = round128(Box::C);  // elements per u stage (128-byte aligned)
  static constexpr int WS = round128(Box::H);  // elements per edge-weight array / stored-u stage
  static constexpr int elems = SC * CS + SP * CS + SW * 3 * WS + SH * WS;
  // Tiles off the FEM block stage only u^k and u^{k-1}: they spend the same
  // shared memory on deeper rings, DP levels ahead.
  static constexpr int deep(int d) { return (d + 4 + pow2(d + 2)) * CS <= elems ? deep(d + 1) : d; }
  static constexpr int DP = deep(D);
  static constexpr int NBX = pow2(DP + 1) > NB ? pow2(DP + 1) : NB;  // barrier pairs allocated
  static constexpr size_t bytes = sizeof(T) * (size_t)elems + 16 * NBX;
};

// Ring sizes of a tile: on the FEM block (all four rings, D levels ahead) or
// off it (DEEP: u^k and u^{k-1} only, DP levels ahead).
template <typename T, bool DEEP>
struct Ring {
  using P = kPipe<T>;
  static constexpr int D = DEEP ? P::DP : P::D;
  static constexpr int SC = D + 3;
  static constexpr int SP = P::pow2(D + 1);
  static constexpr int NB = P::pow2(D + 1);
  static_assert(DEEP ? (SC + SP) * P::CS <= P::elems : (SC == P::SC && SP == P::SP && NB == P::NB), "ring sizes");
};

// Producer side of one interior block: which boxes exist, and their issue.
template <typename T, bool DEEP>
struct Producer {
  const StepArgs<T>* A;
  const Slot<T>* S;
  T *CR, *PR, *WR, *HR;
  uint64_t* full;   // [NB]: the planes of a level have landed (one arrival: the producer, plus bytes)
  uint64_t* empty;  // [NB]: the consumer warps are done with a level (eight arrivals)
  int z0, z1, xf, yf, xw, yw, xh, yh, xp, yp;
  bool fem_tile, hist_tile, pface;  // pface: u^{k-1} with its halo (tiles holding face-adjacent nodes)
  // the planes first read at level g (the first level also reads planes
  // g - 1 and g of u^k, g - 1 of the weights and g of the stored u)
  __device__ __forceinline__ void issue(int g, bool first) const {
    using P = kPipe<T>;
    using R = Ring<T, DEEP>;
    constexpr uint32_t kCBytes = (uint32_t)(Box::C * sizeof(T));
    constexpr uint32_t kPBytes = (uint32_t)(Box::P * sizeof(T));
    constexpr uint32_t kWBytes = (uint32_t)(Box::H * sizeof(T));
    uint64_t* bar = full + ((g - z0) & (R::NB - 1));
    const int wlo = A->wl[2], whi = A->wl[2] + A->wn[2] - 1, hlo = A->fl[2], hhi = A->fh[2];
    const bool c_on = g + 1 <= z1;
    const bool w_on = !DEEP && fem_tile && g >= wlo && g <= whi;
    const bool wm_on = !DEEP && first && fem_tile && g - 1 >= wlo && g - 1 <= whi;
    const bool h_on = !DEEP && hist_tile && g + 1 >= hlo && g + 1 <= hhi;
    const bool h0_on = !DEEP && first && hist_tile && g >= hlo && g <= hhi;
    const uint32_t bytes = kCBytes * ((c_on ? 1 : 0) + (pface ? 1 : 0) + (first ? 2 : 0)) + (pface ? 0u : kPBytes) +
                           kWBytes * (3 * ((w_on ? 1 : 0) + (wm_on ? 1 : 0)) + (h_on ? 1 : 0) + (h0_on ? 1 : 0));
    mbar_arrive_expect_tx(bar, bytes);
    if (first) {
      tma_load_3d(CR + ring<R::SC>(g - 1) * P::CS, &A->tmf, xf, yf, S->zf_cur + g - 1, bar);
      tma_load_3d(CR + ring<R::SC>(g) * P::CS, &A->tmf, xf, yf, S->zf_cur + g, bar);
    }
    if (c_on) tma_load_3d(CR + ring<R::SC>(g + 1) * P::CS, &A->tmf, xf, yf, S->zf_cur + g + 1, bar);
    if (pface)
      tma_load_3d(PR + (g & (R::SP - 1)) * P::CS, &A->tmf, xf, yf, S->zf_prev + g, bar);
    else
      tma_load_3d(PR + (g & (R::SP - 1)) * P::CS, &A->tmp, xp, yp, S->zf_prev + g, bar);
    if (wm_on) weights(g - 1, bar);
    if (w_on) weights(g, bar);
    if (h0_on) tma_load_3d(HR + ring<P::SH>(g) * P::WS, &A->tmh, xh, yh, S->zf_hist + (g - hlo), bar);
    if (h_on) tma_load_3d(HR + ring<P::SH>(g + 1) * P::WS, &A->tmh, xh, yh, S->zf_hist + (g + 1 - hlo), bar);
  }
  // stages and barriers in the block's shared memory, box origins of the
  // tile (i0 - hx, j0 - 1: multiples of 4 in x, so 16-byte aligned)
  __device__ __forceinline__ void setup(const StepArgs<T>& a, const Slot<T>& s, T* sm, uint64_t* bars, int zlo,
                                        int zhi, int i0, int j0, bool hist, bool face) {
    using P = kPipe<T>;
    using R = Ring<T, DEEP>;
    A = &a;
    S = &s;
    CR = sm;
    PR = CR + R::SC * P::CS;
    WR = DEEP ? nullptr : PR + P::SP * P::CS;
    HR = DEEP ? nullptr : WR + P::SW * 3 * P::WS;
    full = bars;
    empty = bars + P::NBX;
    z0 = zlo;
    z1 = zhi;
    xf = i0 - Box::hx;
    yf = j0 - 1;
    xw = i0 - Box::hx - a.wx0;
    yw = j0 - 1 - a.wl[1];
    xh = i0 - Box::hx - a.hx0;
    yh = j0 - a.fl[1];
    xp = i0;
    yp = j0;
    pface = face;
    fem_tile = !DEEP;
    hist_tile = !DEEP && hist;
  }
  __device__ __forceinline__ void weights(int q, uint64_t* bar) const {
    using P = kPipe<T>;
    T* w = WR + ring<P::SW>(q) * 3 * P::WS;
    const int zq = q - A->wl[2];
#pragma unroll
    for (int a = 0; a < 3; ++a) tma_load_3d(w + a * P::WS, &A->tmw, xw, yw, S->zf_w + a * A->wn[2] + zq, bar);
  }
};

// Transposed row with per-axis steps in the gathered order of adj_rhs (diag: the
// coefficient of the node itself).  Its rounding of the diagonal, the same at
// every level, dominates the gradient's FP32 error and is kept: rows from
// differences round better but end up as far from these as both are from FP64.
template <typename T>
__device__ __forceinline__ T gathered_row(T c2, T diag, T wxm, T wxp, T wym, T wyp, T wzm, T wzp, T c, T xm, T xp, T ym,
                                          T yp, T zm, T zp, T pv) {
  T rhs = diag * c;
  rhs += c2 * wxm * xm;
  rhs += c2 * wxp * xp;
  rhs += c2 * wym * ym;
  rhs += c2 * wyp * yp;
  rhs += c2 * wzm * zm;
  rhs += c2 * wzp * zp;
  return rhs - pv;
}

// One node (i, j, k) of an interior block from the staged planes: Ck, Cm, Cp
// are this node in the u^k boxes of planes k, k-1, k+1, Pk in the u^{k-1}
// box, Wk / Wm in the edge-weight arrays of planes k / k-1, Hk / Hp in the
// stored-u boxes of planes k / k+1 (at the voxel origin).  ZF: the plane is
// one step inside a z face (dzs = -1 / +1: the low / high one) and the node
// also produces the face node next to it.  Tiles without FACE hold no node
// one step inside an x or y face.
template <typename T, bool ADJ, bool FEMT, bool FACE, bool ZF, bool REF, bool TEL, bool ANI>
__device__ __forceinline__ void interior_node(const StepArgs<T>& A, const Slot<T>& S, T* __restrict__ gnext,
                                              const Col& C, int k, int off, int dzs, const T* Ck, const T* Cm,
                                              const T* Cp, const T* Pk, const T* Wk, const T* Wm, const T* Hk,
                                              const T* Hp, int rf, T sd) {
  using P = kPipe<T>;
  constexpr int kBoxX = Box::BX;
  if (ZF && FACE && (C.dxs != 0 || C.dys != 0)) return;  // near two faces: edge tiles
  const T c2 = A.c2;
  const T c0 = Ck[0], cm = Cm[0], cp = Cp[0], pv = Pk[0];
  const T xm = Ck[-1], xp = Ck[1], ym = Ck[-kBoxX], yp = Ck[kBoxX];
  bool lf = false;
  const T k0 = ANI ? A.kapt[0] : T(1), k1 = ANI ? A.kapt[1] : T(1), k2 = ANI ? A.kapt[2] : T(1);
  T wxm = k0, wxp = k0, wym = k1, wyp = k1;
  if constexpr (FEMT) lf = C.xy_fem && k >= A.fl[2] && k <= A.fh[2];
  T wzm = k2, wzp = k2;
  T val;
  if (FEMT && lf) {
    wxm = Wk[-1];
    wxp = Wk[0];
    wym = Wk[P::WS - kBoxX];
    wyp = Wk[P::WS];
    wzp = Wk[2 * P::WS];
    wzm = Wm[2 * P::WS];
    const T lap =
        wxp * (xp - c0) + wxm * (xm - c0) + wyp * (yp - c0) + wym * (ym - c0) + wzp * (cp - c0) + wzm * (cm - c0);
    if constexpr (ADJ && ANI)
      val = gathered_row(c2, T(2) + c2 * -(wxp + wxm + wyp + wym + wzp + wzm), wxm, wxp, wym, wyp, wzm, wzp, c0, xm, xp,
                         ym, yp, cm, cp, pv);
    else if constexpr (TEL)  // damped row (sd: the node's damping ratio)
      val = c0 + ((c0 - pv) * (T(1) - sd) + c2 * lap) / (T(1) + sd);
    else
      val = c0 + ((c0 - pv) + c2 * lap);
  } else if constexpr (ADJ && ANI) {
    val = gathered_row(c2, T(2) + c2 * A.kdiag, k0, k0, k1, k1, k2, k2, c0, xm, xp, ym, yp, cm, cp, pv);
  } else if constexpr (ANI) {
    val = c0 + ((c0 - pv) + c2 * ((k0 * ((xm - c0) + (xp - c0)) + k1 * ((ym - c0) + (yp - c0))) +
                                  k2 * ((cm - c0) + (cp - c0))));
  } else {  // unit weights: the neighbour sum minus 6 u^k
    val = c0 + ((c0 - pv) + c2 * ((((xm + xp) + (ym + yp)) + (cm + cp)) - T(6) * c0));
  }
  if constexpr (ZF) {  // the z face node next to this node (the rows of the x / y faces below)
    const int f = dzs > 0 ? 5 : 4;
    const T* Cb = dzs > 0 ? Cp : Cm;  // b and its in-face neighbours in the staged plane k +- 1
    const T ub = Cb[0];
    const bool abc = (S.mask_f >> f) & 1;
    const int offb = off + dzs * A.px * A.ny;
    const long long gb = (gnext - S.next) + offb;  // (fields hold 2^31 nodes and more; an item's offsets fit 32 bits)
    const T rf = ANI ? A.ra[2] : A.r;
    if constexpr (!ADJ) {
      T vb;
      if (abc) {
        vb = rf * ub + (c0 - rf * val);
      } else {
        T lb = T(2) * k2 * (c0 - ub);
        lb += k0 * ((Cb[-1] - ub) + (Cb[1] - ub));
        lb += k1 * ((Cb[-kBoxX] - ub) + (Cb[kBoxX] - ub));
        vb = ub + ((ub - S.prev[gb]) + c2 * lb);  // (u^{k-1} of the face plane is not staged)
        if ((S.src_mask >> f) & 1) vb += src_term(S, f, C.i, C.j, k + dzs);
        if (S.inj && S.obs_face == f) vb += S.inj_scale * T(2) * S.inj[face_index(f, C.i, C.j, k + dzs, A.nx, A.ny)];
      }
      gnext[offb] = vb;
      if (S.obs_w && S.obs_face == f) S.obs_w[face_index(f, C.i, C.j, k + dzs, A.nx, A.ny)] = vb;
    } else {
      const T coef_mb = dzs > 0 ? wzp : wzm;
      T lb = abc ? rf * ub : (ANI ? T(2) + c2 * A.kdiag : T(2) - T(6) * c2) * ub;
      lb += c2 * coef_mb * c0;
      if (!abc) {
        lb += c2 * k0 * (Cb[-1] + Cb[1]);
        lb += c2 * k1 * (Cb[-kBoxX] + Cb[kBoxX]);
      }
      if (!((S.mask_c >> f) & 1)) lb -= S.prev[gb];
      if (S.obs_r && S.obs_face == f) lb += S.obs_r[face_index(f, C.i, C.j, k + dzs, A.nx, A.ny)];
      val += (abc ? ub : T(2) * c2 * k2 * ub) - c2 * coef_mb * ub;
      if ((S.mask_e >> f) & 1) val -= rf * lb;
      gnext[offb] = lb;
    }
  }
  if constexpr (FACE) {
    if (C.dxs != 0 || C.dys != 0) {  // the x or y face node next to this node
      const int ax = C.dxs ? 0 : 1;
      const int sd = C.dxs ? C.dxs : C.dys;
      const int f = 2 * ax + (sd > 0 ? 1 : 0);
      const int ob = ax == 0 ? sd : sd * kBoxX;  // b relative to this node in a u box
      const int o1 = ax == 0 ? kBoxX : 1;        // the other in-plane axis in the box
      const T ub = Ck[ob];
      const bool abc = (S.mask_f >> f) & 1;
      const int offb = off + (ax == 0 ? sd : sd * A.px);
      const int bi = C.i + (ax == 0 ? sd : 0), bj = C.j + (ax == 1 ? sd : 0);
      const T rf = ANI ? A.ra[ax] : A.r, kn = ax == 0 ? k0 : k1, kt = ax == 0 ? k1 : k0;  // across, along the face
      // Forward: the absorbing row of Eq. (eq:abs2) from u^k at b and m and
      // the new value at m, or the mirror-ghost row with the source flux.
      // Transposed: b's row in closed form (no transposed absorbing coupling
      // reaches it), from lambda^{j+1} at b and m, the coefficient of m's row
      // on b and lambda^{j+2} at b.  The in-face neighbours (the other
      // in-plane axis first, then z) are read only for non-absorbing faces.
      if constexpr (!ADJ) {
        T vb;
        if (abc) {
          vb = rf * ub + (c0 - rf * val);
        } else {
          T lb = T(2) * kn * (c0 - ub);
          lb += kt * ((Ck[ob - o1] - ub) + (Ck[ob + o1] - ub));
          lb += k2 * ((Cm[ob] - ub) + (Cp[ob] - ub));
          vb = ub + ((ub - Pk[ob]) + c2 * lb);
          if ((S.src_mask >> f) & 1) vb += src_term(S, f, bi, bj, k);
          if (S.inj && S.obs_face == f) vb += S.inj_scale * T(2) * S.inj[face_index(f, bi, bj, k, A.nx, A.ny)];
        }
        gnext[offb] = vb;
        if (S.obs_w && S.obs_face == f) S.obs_w[face_index(f, bi, bj, k, A.nx, A.ny)] = vb;
      } else {
        const T coef_mb = ax == 0 ? (sd > 0 ? wxp : wxm) : (sd > 0 ? wyp : wym);
        T lb = abc ? rf * ub : (ANI ? T(2) + c2 * A.kdiag : T(2) - T(6) * c2) * ub;
        lb += c2 * coef_mb * c0;
        if (!abc) {
          lb += c2 * kt * (Ck[ob - o1] + Ck[ob + o1]);
          lb += c2 * k2 * (Cm[ob] + Cp[ob]);
        }
        if (!((S.mask_c >> f) & 1)) lb -= Pk[ob];
        if (S.obs_r && S.obs_face == f) lb += S.obs_r[face_index(f, bi, bj, k, A.nx, A.ny)];
        val += (abc ? ub : T(2) * c2 * kn * ub) - c2 * coef_mb * ub;
        if ((S.mask_e >> f) & 1) val -= rf * lb;
        gnext[offb] = lb;
      }
    }
  }
  if (!(FEMT && lf)) {
    gnext[off] = val;
    return;
  }
  const int bo = (C.i - A.hx0) + A.hpx * ((C.j - A.fl[1]) + A.fn[1] * (k - A.fl[2]));
  // rf: the node's refinement flags (0 off the columns' refined z ranges)
  if (!(REF && (rf & 1))) {  // (the refined rows write those)
    gnext[off] = val;
    if (!ADJ && S.hist_w) S.hist_w[bo] = TEL ? val - pv : val;  // (telegraph: u^{k+1} - u^{k-1})
  }
  if constexpr (ADJ) {
    const int vz = A.un[0] * A.un[1];
    const int vid = (C.i - A.fl[0]) + A.un[0] * (C.j - A.fl[1]) + vz * (k - A.fl[2]);
    if (C.xy_vox && k < A.fl[2] + A.un[2] && !(REF && (rf & 2))) {
      const T u[8] = {Hk[0], Hk[1], Hk[kBoxX], Hk[kBoxX + 1], Hp[0], Hp[1], Hp[kBoxX], Hp[kBoxX + 1]};
      const T l[8] = {c0, xp, yp, Ck[kBoxX + 1], cp, Cp[1], Cp[kBoxX], Cp[kBoxX + 1]};
      atomicAdd(A.G + (long long)C.si * ((long long)vz * A.un[2]) + vid, (double)(TEL ? damp_sum(u, l) : (ANI ? pair_sum_ani(A, u, l) : pair_sum(u, l))));
    }
  }
}

// The x face column of a tile whose lanes would otherwise diverge: lanes 1
// .. 16 of the producer warp, one tile row each, compute the node m one step
// inside the face (off the FEM block: unit weights) and the face node b next
// to it, so that the consumer warps skip m.  Planes and rows next to another
// face belong to the edge tiles.  The rows are those of interior_node.
struct XFace {
  bool on;   // the tile uses the face lanes
  int mi;    // x of the nodes m (1 or nx - 2)
  int sd;    // -1 / +1: the low / high x face
  int i0, j0;
};
constexpr unsigned kFaceLanes = 0x1fffeu;  // lanes 1 .. 16 of the producer warp

template <typename T, bool ADJ, bool DEEP, bool ANI>
__device__ __forceinline__ void xface_levels(const StepArgs<T>& A, const Slot<T>& S, const Producer<T, DEEP>& pr,
                                             const XFace& X, int z0, int z1, long long budget) {
  using P = kPipe<T>;
  using R = Ring<T, DEEP>;
  const int r = (int)threadIdx.x - (kTileX * kTileY / 2 + 1);  // tile row 0 .. 15
  const int j = X.j0 + r;
  const bool row_on = j >= 2 && j <= A.ny - 3;
  const int f = X.sd > 0 ? 1 : 0;
  const int sd = X.sd;
  constexpr int kBoxX = Box::BX;
  const int o = (r + 1) * kBoxX + (X.mi - X.i0 + Box::hx);  // m in a u box
  const T c2 = A.c2, rf = ANI ? A.ra[0] : A.r;
  const T k0 = ANI ? A.kapt[0] : T(1), k1 = ANI ? A.kapt[1] : T(1), k2 = ANI ? A.kapt[2] : T(1);
  const bool abc = (S.mask_f >> f) & 1;
  const int pl = A.px * A.ny;
  T* __restrict__ gnext = S.next + (long long)pl * z0;
  int off = X.mi + A.px * j;
  for (int k = z0; k < z1; ++k, off += pl) {
    const int q = k - z0;
    const bool ok = mbar_wait(pr.full + (q & (R::NB - 1)), (uint32_t)((q / R::NB) & 1), budget, A.err);
    if (!__all_sync(kFaceLanes, ok)) {
      if (r == 0) atomicExch(A.err, 1);
      return;
    }
    if (row_on && k >= 2 && k <= A.nz - 3) {
      const T* Ck = pr.CR + ring<R::SC>(k) * P::CS + o;
      const T* Cm = pr.CR + ring<R::SC>(k - 1) * P::CS + o;
      const T* Cp = pr.CR + ring<R::SC>(k + 1) * P::CS + o;
      const T* Pk = pr.PR + (k & (R::SP - 1)) * P::CS + o;
      const T c0 = Ck[0], xm = Ck[-1], xp = Ck[1], ym = Ck[-kBoxX], yp = Ck[kBoxX];
      const T cm = Cm[0], cp = Cp[0], pv = Pk[0];
      T val;
      if constexpr (ADJ && ANI)
        val = gathered_row(c2, T(2) + c2 * A.kdiag, k0, k0, k1, k1, k2, k2, c0, xm, xp, ym, yp, cm, cp, pv);
      else if constexpr (ANI)
        val = c0 + ((c0 - pv) + c2 * ((k0 * ((xm - c0) + (xp - c0)) + k1 * ((ym - c0) + (yp - c0))) +
                                      k2 * ((cm - c0) + (cp - c0))));
      else
        val = c0 + ((c0 - pv) + c2 * ((((xm + xp) + (ym + yp)) + (cm + cp)) - T(6) * c0));
      const T ub = Ck[sd];
      const int offb = off + sd;
      if constexpr (!ADJ) {
        T vb;
        if (abc) {
          vb = rf * ub + (c0 - rf * val);
        } else {
          T lb = T(2) * k0 * (c0 - ub);
          lb += k1 * ((Ck[sd - kBoxX] - ub) + (Ck[sd + kBoxX] - ub));
          lb += k2 * ((Cm[sd] - ub) + (Cp[sd] - ub));
          vb = ub + ((ub - Pk[sd]) + c2 * lb);
          if ((S.src_mask >> f) & 1) vb += src_term(S, f, X.mi + sd, j, k);
          if (S.inj && S.obs_face == f) vb += S.inj_scale * T(2) * S.inj[face_index(f, X.mi + sd, j, k, A.nx, A.ny)];
        }
        gnext[offb] = vb;
        if (S.obs_w && S.obs_face == f) S.obs_w[face_index(f, X.mi + sd, j, k, A.nx, A.ny)] = vb;
      } else {
        T lb = abc ? rf * ub : (ANI ? T(2) + c2 * A.kdiag : T(2) - T(6) * c2) * ub;
        lb += c2 * k0 * c0;
        if (!abc) {
          lb += c2 * k1 * (Ck[sd - kBoxX] + Ck[sd + kBoxX]);
          lb += c2 * k2 * (Cm[sd] + Cp[sd]);
        }
        if (!((S.mask_c >> f) & 1)) lb -= Pk[sd];
        if (S.obs_r && S.obs_face == f) lb += S.obs_r[face_index(f, X.mi + sd, j, k, A.nx, A.ny)];
        val += (abc ? ub : T(2) * c2 * k0 * ub) - c2 * k0 * ub;
        if ((S.mask_e >> f) & 1) val -= rf * lb;
        gnext[offb] = lb;
      }
      gnext[off] = val;
    }
    __syncwarp(kFaceLanes);  // the lanes' reads of level k's stages are done
    if (r == 0) mbar_arrive(pr.empty + (q & (R::NB - 1)));
  }
}

// Consumer loop of an interior block, specialised by whether the tile meets
// the FEM block (FEMT) and whether it holds nodes one step inside an x or y
// face (FACE).  Each consumer thread owns two tile rows (ty and ty + 8).
template <typename T, bool ADJ, bool FEMT, bool FACE, bool REF, bool TEL, bool ANI>
__device__ __forceinline__ void interior_levels(const StepArgs<T>& A, const Slot<T>& S, const Col (&C)[2],
                                                const Producer<T, !FEMT>& pr, const bool (&active)[2],
                                                const XFace& X, int z0, int z1) {
  using P = kPipe<T>;
  using R = Ring<T, !FEMT>;
  constexpr int D = R::D;
  constexpr int kProd = kTileX * kTileY / 2;  // the producer thread
  const int t = (int)threadIdx.x;
  const long long budget = A.wait;            // cycles a pipeline wait may take
  if (t >= kProd) {
    // Producer: the planes first read at level g overwrite stages last read
    // at level g - D - 1 (the edge-weight and stored-u rings are the
    // shortest), so they are issued once every consumer warp is done with it.
    if (t != kProd) {
      if (FACE && X.on && t <= kProd + 16) xface_levels<T, ADJ, !FEMT, ANI>(A, S, pr, X, z0, z1, budget);
      return;
    }
    for (int g = 0; g < D && z0 + g < z1; ++g) pr.issue(z0 + g, g == 0);
    int g = z0 + D;
    for (; g < z1; ++g) {
      const int q = g - D - 1 - z0;
      if (q >= 0 && !mbar_wait(pr.empty + (q & (R::NB - 1)), (uint32_t)((q / R::NB) & 1), budget, A.err)) {
        atomicExch(A.err, 1);
        break;
      }
      fence_proxy_async_shared();
      pr.issue(g, false);
    }
    // let no copy be in flight when the block exits (the consumers may have
    // given up): wait for the last issued levels, ignoring the abort flag and
    // the pipeline's own limit (the copies complete within microseconds)
    const int no_abort = 0;
    const int issued = min(g, z1) - z0;
    for (int q = max(0, issued - R::NB); q < issued; ++q)
      mbar_wait(pr.full + (q & (R::NB - 1)), (uint32_t)((q / R::NB) & 1), kDrainCycles, &no_abort);
    return;
  }
  // Consumers: each warp waits for level k's planes, computes its nodes and
  // releases the level; warps run up to D levels apart.
  const int tx = t & 31, ty = t >> 5;
  const int nz = A.nz;
  const int pl = A.px * A.ny;
  constexpr int kBoxX = Box::BX;
  const int o0 = (ty + 1) * kBoxX + (tx + Box::hx);  // row 0 in a u box / edge-weight array
  const int o1 = o0 + (kTileY / 2) * kBoxX;             // row 1
  const int h0 = ty * kBoxX + (tx + Box::hx);        // row 0 in a stored-u box
  const int h1 = h0 + (kTileY / 2) * kBoxX;
  // u^{k-1}: the u box layout on face tiles, else the halo-free box
  const int p0 = FACE ? o0 : ty * Box::PX + tx;
  const int p1 = FACE ? o1 : p0 + (kTileY / 2) * Box::PX;
  const bool act0 = !FACE || active[0], act1 = !FACE || active[1];  // every row of a tile off the faces is active
  T* __restrict__ gnext = S.next + (long long)pl * z0;
  int off0 = C[0].i + A.px * C[0].j;                 // field offsets of the two nodes from plane z0
  int off1 = off0 + (kTileY / 2) * A.px;
  // refinement flags of the two nodes, loaded one level ahead (their
  // latency then overlaps the wait for the level's planes)
  auto rflag = [&](const Col& c, int kk) -> int {
    if (!REF || kk < c.rz0 || kk > c.rz1) return 0;
    return A.rmask[(c.i - A.hx0) + A.hpx * ((c.j - A.fl[1]) + A.fn[1] * (kk - A.fl[2]))];
  };
  int rfn0 = 0, rfn1 = 0;
  if constexpr (REF) {
    rfn0 = rflag(C[0], z0);
    rfn1 = rflag(C[1], z0);
  }
  // telegraph reading: the nodes' damping ratios, likewise a level ahead
  auto sdamp = [&](const Col& c, int kk) -> T {
    if (!TEL || !c.xy_fem || kk < A.fl[2] || kk > A.fh[2]) return T(0);
    return A.sdamp[(c.i - A.hx0) + A.hpx * ((c.j - A.fl[1]) + A.fn[1] * (kk - A.fl[2]))];
  };
  T sdn0 = T(0), sdn1 = T(0);
  if constexpr (TEL) {
    sdn0 = sdamp(C[0], z0);
    sdn1 = sdamp(C[1], z0);
  }
  // ring stages of planes k - 1, k, k + 1 (rotated from level to level
  // instead of reduced modulo the ring size at every level)
  int scm = ring<R::SC>(z0 - 1), sck = ring<R::SC>(z0), scp = ring<R::SC>(z0 + 1);
  int swm = 0, swk = 0, shk = 0, shp = 0;
  if constexpr (FEMT) {
    swm = ring<P::SW>(z0 - 1);
    swk = ring<P::SW>(z0);
    shk = ring<P::SH>(z0);
    shp = ring<P::SH>(z0 + 1);
  }
  for (int k = z0; k < z1; ++k, off0 += pl, off1 += pl) {
    const int q = k - z0;
    const int rf0 = rfn0, rf1 = rfn1;
    if constexpr (REF) {
      if (k + 1 < z1) {
        rfn0 = rflag(C[0], k + 1);
        rfn1 = rflag(C[1], k + 1);
      }
    }
    const T sd0 = sdn0, sd1 = sdn1;
    if constexpr (TEL) {
      if (k + 1 < z1) {
        sdn0 = sdamp(C[0], k + 1);
        sdn1 = sdamp(C[1], k + 1);
      }
    }
    const bool ok = mbar_wait(pr.full + (q & (R::NB - 1)), (uint32_t)((q / R::NB) & 1), budget, A.err);
    if (!__all_sync(0xffffffffu, ok)) {
      if (tx == 0) atomicExch(A.err, 1);
      return;
    }
    const T* Ck = pr.CR + sck * P::CS;
    const T* Cm = pr.CR + scm * P::CS;
    const T* Cp = pr.CR + scp * P::CS;
    const T* Pk = pr.PR + (k & (R::SP - 1)) * P::CS;
    const T* Wk = nullptr;
    const T* Wm = nullptr;
    const T* Hk = nullptr;
    const T* Hp = nullptr;
    if constexpr (FEMT) {
      Wk = pr.WR + swk * 3 * P::WS;
      Wm = pr.WR + swm * 3 * P::WS;
      Hk = pr.HR + shk * P::WS;
      Hp = pr.HR + shp * P::WS;
    }
    // planes one step inside a z face also produce the face plane (block-uniform)
    const int dzs = k == 1 ? -1 : (k == nz - 2 ? 1 : 0);
    if (dzs != 0) {
      if (act0)
        interior_node<T, ADJ, FEMT, FACE, true, REF, TEL, ANI>(A, S, gnext, C[0], k, off0, dzs, Ck + o0, Cm + o0, Cp + o0,
                                                Pk + p0, Wk + o0, Wm + o0, Hk + h0, Hp + h0, rf0, sd0);
      if (act1)
        interior_node<T, ADJ, FEMT, FACE, true, REF, TEL, ANI>(A, S, gnext, C[1], k, off1, dzs, Ck + o1, Cm + o1, Cp + o1,
                                                Pk + p1, Wk + o1, Wm + o1, Hk + h1, Hp + h1, rf1, sd1);
    } else {
      if (act0)
        interior_node<T, ADJ, FEMT, FACE, false, REF, TEL, ANI>(A, S, gnext, C[0], k, off0, 0, Ck + o0, Cm + o0, Cp + o0,
                                                 Pk + p0, Wk + o0, Wm + o0, Hk + h0, Hp + h0, rf0, sd0);
      if (act1)
        interior_node<T, ADJ, FEMT, FACE, false, REF, TEL, ANI>(A, S, gnext, C[1], k, off1, 0, Ck + o1, Cm + o1, Cp + o1,
                                                 Pk + p1, Wk + o1, Wm + o1, Hk + h1, Hp + h1, rf1, sd1);
    }
    __syncwarp();  // the warp's reads of level k's stages are done
    if (tx == 0) mbar_arrive(pr.empty + (q & (R::NB - 1)));
    scm = sck;
    sck = scp;
    scp = scp + 1 == R::SC ? 0 : scp + 1;
    if constexpr (FEMT) {
      swm = swk;
      swk = swk + 1 == P::SW ? 0 : swk + 1;
      shk = shp;
      shp = shp + 1 == P::SH ? 0 : shp + 1;
    }
  }
}

// Interior part of one time level (lattices with >= 5 nodes per axis):
// 32 x 16 tiles of the nodes 1 .. n-2 and z ranges, one block per work item
// (slot, tile, z range; the host balances the items by cost): eight
// consumer warps (two tile rows per thread) and a producer warp.  Nodes one
// step inside a face also produce the face node next to them.
template <typename T, bool ADJ, bool TEL, bool ANI>
__device__ __forceinline__ void interior_block(const StepArgs<T>& A, int b, T* sm) {
  static_assert(kTileX == 32, "one warp per tile row");
  static_assert(kTileX * kTileY / 2 + 32 == kStepBlock, "eight consumer warps (two rows each) and a producer warp");
  using P = kPipe<T>;
  const int* item = A.items + 4 * b;  // (slot, tile, z0, z1)
  const int si = item[0];
  const int tyy = item[1] / A.ntx;
  const int txx = item[1] - tyy * A.ntx;
  const int z0 = item[2], z1 = item[3];
  const int nx = A.nx, ny = A.ny;
  if (z0 >= z1) return;  // whole block
  const int t = (int)threadIdx.x;
  const int tx = t & 31, ty = t >> 5;
  const int i0 = txx * kTileX, j0 = 1 + tyy * kTileY;
  const Slot<T>& S = A.s[si];
  const bool has_fem = A.fl[0] <= A.fh[0];
  const bool pairing = ADJ && S.hist_r != nullptr;
  Col C[2];
  bool active[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    C[r].si = si;
    C[r].i = i0 + tx;
    C[r].j = j0 + ty + r * (kTileY / 2);
    C[r].dxs = (C[r].i == 1) ? -1 : (C[r].i == nx - 2 ? 1 : 0);
    C[r].dys = (C[r].j == 1) ? -1 : (C[r].j == ny - 2 ? 1 : 0);
    active[r] = t < kTileX * kTileY / 2 && C[r].i >= 1 && C[r].i <= nx - 2 && C[r].j <= ny - 2 &&
                !(C[r].dxs != 0 && C[r].dys != 0);
    C[r].xy_fem = has_fem && C[r].i >= A.fl[0] && C[r].i <= A.fh[0] && C[r].j >= A.fl[1] && C[r].j <= A.fh[1];
    C[r].xy_uv = has_fem && C[r].i >= A.fl[0] && C[r].i < A.fl[0] + A.un[0] && C[r].j >= A.fl[1] &&
                 C[r].j < A.fl[1] + A.un[1];
    C[r].xy_vox = pairing && C[r].xy_uv;
    C[r].rz0 = 1;
    C[r].rz1 = 0;
    if (A.rzr && C[r].xy_fem) {
      const int c = (C[r].i - A.fl[0]) + A.fn[0] * (C[r].j - A.fl[1]);
      C[r].rz0 = A.rzr[2 * c];
      C[r].rz1 = A.rzr[2 * c + 1];
    }
  }
  // x face column handled by the face lanes: one x face in the tile, and
  // its column m off the FEM block
  XFace X;
  {
    const bool xlo = i0 <= 1, xhi = i0 + kTileX - 1 >= nx - 2;  // the tile holds node 1 / node nx - 2
    X.mi = xlo ? 1 : nx - 2;
    X.sd = xlo ? -1 : 1;
    X.i0 = i0;
    X.j0 = j0;
    X.on = xlo != xhi && !(has_fem && X.mi >= A.fl[0] && X.mi <= A.fh[0]);
    if (X.on) {
      active[0] = active[0] && C[0].dxs == 0;
      active[1] = active[1] && C[1].dxs == 0;
    }
  }
  // block-uniform tile kinds: an item whose planes hold no FEM-owned node
  // needs no edge weights or history and runs with the deep rings
  const bool fem_tile = has_fem && i0 <= A.fh[0] && i0 + kTileX - 1 >= A.fl[0] && j0 <= A.fh[1] &&
                        j0 + kTileY - 1 >= A.fl[1] && z0 <= A.fh[2] && z1 - 1 >= A.fl[2];
  const bool face_tile = i0 <= 1 || i0 + kTileX - 1 >= nx - 2 || j0 == 1 || j0 + kTileY - 1 >= ny - 2;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + P::elems);
  const int tp = kTileX * kTileY / 2;  // the producer thread
  if (t == tp) {
    for (int q = 0; q < P::NBX; ++q) {
      mbar_init(full + q, 1);
      mbar_init(full + P::NBX + q, kTileX * kTileY / 2 / 32 + (X.on ? 1 : 0));  // consumer warps (+ face lanes)
    }
    mbar_init_fence();
  }
  pdl_wait();  // the previous level is complete: its output may be read, its input overwritten
  __syncthreads();
  // items whose columns hold refined-voxel corners in their z range take the
  // variant with the refined rows (block-uniform)
  const bool ref_tile =
      __syncthreads_or(fem_tile && t < kTileX * kTileY / 2 &&
                       ((C[0].rz0 <= C[0].rz1 && C[0].rz0 < z1 && C[0].rz1 >= z0) ||
                        (C[1].rz0 <= C[1].rz1 && C[1].rz0 < z1 && C[1].rz1 >= z0)));
  if (fem_tile) {
    Producer<T, false> pr;
    pr.setup(A, S, sm, full, z0, z1, i0, j0, pairing, face_tile);
    if constexpr (TEL) {  // telegraph reading (no refinement)
      if (face_tile)
        interior_levels<T, ADJ, true, true, false, true, false>(A, S, C, pr, active, X, z0, z1);
      else
        interior_levels<T, ADJ, true, false, false, true, false>(A, S, C, pr, active, X, z0, z1);
    } else if (!ANI && ref_tile) {  // (no refinement with per-axis steps)
      if (face_tile)
        interior_levels<T, ADJ, true, true, !ANI, false, ANI>(A, S, C, pr, active, X, z0, z1);
      else
        interior_levels<T, ADJ, true, false, !ANI, false, ANI>(A, S, C, pr, active, X, z0, z1);
    } else {
      if (face_tile)
        interior_levels<T, ADJ, true, true, false, false, ANI>(A, S, C, pr, active, X, z0, z1);
      else
        interior_levels<T, ADJ, true, false, false, false, ANI>(A, S, C, pr, active, X, z0, z1);
    }
  } else {
    Producer<T, true> pr;
    pr.setup(A, S, sm, full, z0, z1, i0, j0, false, face_tile);
    if (face_tile)
      interior_levels<T, ADJ, false, true, false, false, ANI>(A, S, C, pr, active, X, z0, z1);
    else
      interior_levels<T, ADJ, false, false, false, false, ANI>(A, S, C, pr, active, X, z0, z1);
  }
}

// Edge tile of the forward step.  Levels by the number of faces a node lies
// on: nodes on no face take their interior row, then face, edge and corner
// nodes; an absorbing row (Eq. (eq:abs2)) reads the new values of its
// inward neighbours, one level down in the same tile, from shared memory.
// Every thread of the block calls it (it synchronises); nv holds 128 values.
template <typename T, bool ANI>
__device__ __forceinline__ void fwd_edge_tile(const StepArgs<T>& A, int si, int blk, int t, T* nv) {
  const Slot<T>& S = A.s[si];
  int i = 0, j = 0, k = 0, nf = -1, q[3];
  const bool valid = blk < A.nedge && edge_tile_node(A, blk, t, i, j, k, q, nf);
  const long long id = valid ? lin(A, i, j, k) : 0;
  const int fall = valid ? face_bits(i, j, k, A.nx, A.ny, A.nz) : 0;
  const int fb = fall & S.mask_f;
  // u^k at the node and at its inward neighbour across each absorbing face,
  // loaded before the levels below (which then wait only on shared memory)
  const T cself = valid ? S.cur[id] : T(0);
  T cin[3];
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int fa = (fb >> (2 * ax)) & 3;
    cin[ax] = (valid && fa) ? S.cur[id + ((fa & 1) ? 1 : -1) * axis_stride(A, ax)] : T(0);
  }
  T plain = T(0);  // the non-absorbing row, from level-k data only
  if (valid && !fb) {
    plain = cself + ((cself - S.prev[id]) + A.c2 * row_lap_inl<T, ANI>(A, S.W, S.cur, i, j, k));
    if (fall & S.src_mask) plain += src_terms(S, fall, i, j, k);
    if (S.inj) plain += inj_term(S, fall, i, j, k, A.nx, A.ny);
  }
  nv[t] = plain;
  __syncthreads();
  for (int level = 1; level <= 3; ++level) {
    T v = T(0);
    const bool mine = valid && fb && __popc(fall) == level;
    if (mine) {
      T acc = T(0);
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const int fa = (fb >> (2 * ax)) & 3;
        if (!fa) continue;
        const int t1 = edge_tile_peer(t, blk, q, ax, (fa & 1) ? 1 : 2);
        acc += cin[ax] - (ANI ? A.ra[ax] : A.r) * nv[t1];
      }
      v = (ANI ? abc_self(A, fb) : A.r) * cself + acc / T(__popc(fb));
    }
    __syncthreads();
    if (mine) nv[t] = v;
    __syncthreads();
  }
  if (!valid) return;
  const T val = nv[t];
  S.next[id] = val;
  if (S.obs_w && ((fall >> S.obs_face) & 1)) S.obs_w[face_index(S.obs_face, i, j, k, A.nx, A.ny)] = val;
  if (S.hist_w && fem_owned(A, i, j, k)) S.hist_w[hidx(A, i, j, k)] = val;
}

// Edge tile of the transposed step: every thread gathers its transposed row
// in parallel, then the transposed absorbing couplings (E^T) are resolved
// from the nodes on the most faces inwards, through shared memory.
template <typename T, bool ANI>
__device__ __forceinline__ void adj_edge_tile(const StepArgs<T>& A, int si, int blk, int t, T* lam) {
  const Slot<T>& S = A.s[si];
  int i = 0, j = 0, k = 0, nf = -1, q[3];
  const bool valid = blk < A.nedge && edge_tile_node(A, blk, t, i, j, k, q, nf);
  lam[t] = valid ? adj_rhs_inl<T, ANI>(A, S, i, j, k) : T(0);
  __syncthreads();
  for (int level = 2; level >= 0; --level) {
    T v = T(0);
    const bool mine = valid && nf == level;
    if (mine) {
      v = lam[t];
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        if (q[ax] != 1 && q[ax] != 2) continue;  // not one node inside a face on this axis
        const int s = q[ax] == 1 ? -1 : 1;
        const int bi = i + (ax == 0 ? s : 0), bj = j + (ax == 1 ? s : 0), bk = k + (ax == 2 ? s : 0);
        const int f = 2 * ax + (s > 0 ? 1 : 0);
        const int fbb = face_bits(bi, bj, bk, A.nx, A.ny, A.nz) & S.mask_e;
        if (!(fbb & (1 << f))) continue;
        v -= ((ANI ? A.ra[ax] : A.r) / T(__popc(fbb))) * lam[edge_tile_peer(t, blk, q, ax, q[ax] == 1 ? 0 : 3)];
      }
    }
    __syncthreads();
    if (mine) lam[t] = v;
    __syncthreads();
  }
  if (!valid) return;
  S.next[lin(A, i, j, k)] = lam[t];
  pair_if_voxel<T, ANI>(A, S, si, i, j, k);
}

template <typename T, bool ADJ>
__device__ __forceinline__ void refined_rows(const StepArgs<T>& A, long long t);
template <typename T>
__device__ __noinline__ void paper_voxels(const StepArgs<T>& A, long long t);

// One time level of every slot in one launch of kStepBlock threads per
// block: first the edge tiles (two 128-node tiles per block, so their short
// dependent chains start early), then the interior blocks, then the rows of
// the refined region (gathers of short latency-bound rows, which fill the
// slots the interior blocks free towards the end of the level), and in the
// paper's adjoint the pairing of the unknown voxels.  All blocks
// read levels k, k-1 and write disjoint nodes of level k+1.
// (PAIR: the paper's adjoint with a history to pair with, a variant of its own,
// as the forward levels lose 1 - 2 % to the mere presence of that branch.)
template <typename T, bool ADJ, bool TEL, bool ANI, bool PAIR = false>
__global__ void __launch_bounds__(kStepBlock, 4) step_kernel(const __grid_constant__ StepArgs<T> A) {
  extern __shared__ __align__(128) unsigned char hyb_smem[];  // kPipe<T>::bytes
  T* sh = reinterpret_cast<T*>(hyb_smem);
  pdl_trigger();  // the next level's launch may start its blocks
  int b = blockIdx.x;
  if (b < A.nhe) {  // two 128-node tiles; the last warp takes part in the barriers only
    pdl_wait();     // the previous level is complete
    const int ne2 = (A.nedge + 1) / 2;
    const int si = b / ne2;
    const int half = (int)(threadIdx.x >> 7);
    const int blk = half < 2 ? 2 * (b - si * ne2) + half : A.nedge;
    const int t = (int)(threadIdx.x & 127);
    if constexpr (ADJ)
      adj_edge_tile<T, ANI>(A, si, blk, t, sh + 128 * half);
    else
      fwd_edge_tile<T, ANI>(A, si, blk, t, sh + 128 * half);
    return;
  }
  b -= A.nhe;
  if (b >= A.nitems) {
    pdl_wait();
    b -= A.nitems;
    if constexpr (PAIR)
      if (b >= A.nhr) {
        paper_voxels(A, (long long)(b - A.nhr) * kStepBlock + threadIdx.x);
        return;
      }
    if constexpr (!ANI) refined_rows<T, ADJ>(A, (long long)b * kStepBlock + threadIdx.x);
    return;
  }
  interior_block<T, ADJ, TEL, ANI>(A, b, sh);
}

// Lattices with fewer than 5 nodes on some axis: every node by the generic
// rows (forward and transposed).
template <typename T>
__global__ void __launch_bounds__(128) fwd_all_kernel(const __grid_constant__ StepArgs<T> A) {
  const long long n = (long long)A.nx * A.ny * A.nz;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * A.nslots) return;
  const int si = (int)(t / n);
  const long long q = t - (long long)si * n;
  const int i = (int)(q % A.nx);
  const int j = (int)((q / A.nx) % A.ny);
  const int k = (int)(q / ((long long)A.nx * A.ny));
  const long long id = lin(A, i, j, k);
  const Slot<T>& S = A.s[si];
  const T val = fwd_new<T, 3>(A, S, i, j, k);
  S.next[id] = val;
  if (S.obs_w && ((face_bits(i, j, k, A.nx, A.ny, A.nz) >> S.obs_face) & 1))
    S.obs_w[face_index(S.obs_face, i, j, k, A.nx, A.ny)] = val;
  if (S.hist_w && fem_owned(A, i, j, k)) S.hist_w[hidx(A, i, j, k)] = val;
}

template <typename T>
__global__ void __launch_bounds__(128) adj_all_kernel(const __grid_constant__ StepArgs<T> A) {
  const long long n = (long long)A.nx * A.ny * A.nz;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * A.nslots) return;
  const int si = (int)(t / n);
  const long long q = t - (long long)si * n;
  const int i = (int)(q % A.nx);
  const int j = (int)((q / A.nx) % A.ny);
  const int k = (int)(q / ((long long)A.nx * A.ny));
  const Slot<T>& S = A.s[si];
  S.next[lin(A, i, j, k)] = adj_new<T, 3>(A, S, i, j, k);
  pair_if_voxel<T, true>(A, S, si, i, j, k);
}

template <typename T>
__global__ void pair_kernel(const __grid_constant__ StepArgs<T> A, const T* __restrict__ hist,
                            const T* __restrict__ lam, double* __restrict__ grad) {
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nv) return;
  const int x = (int)(t % A.un[0]);
  const long long r = t / A.un[0];
  const int y = (int)(r % A.un[1]);
  const int z = (int)(r / A.un[1]);
  if (A.refvox && A.refvox[t]) return;
  const int i = A.fl[0] + x, j = A.fl[1] + y, k = A.fl[2] + z;
  grad[t] += (double)(A.tet ? tet_pair(A, hist, lam, i, j, k)
                             : (A.ani ? voxel_pair_ani(A, hist, lam, i, j, k) : voxel_pair(A, hist, lam, i, j, k)));
}

// Threads of the refined trailing blocks, per slot: the corner rows, then
// the centre rows (with the transposed step's pairing of their voxels).
template <typename T, bool ADJ>
__device__ __forceinline__ void refined_rows(const StepArgs<T>& A, long long t) {
  const int per = A.nrl + A.nref;
  if (t >= (long long)per * A.nslots) return;
  const int si = (int)(t / per);
  const int r = (int)(t - (long long)si * per);
  const Slot<T>& S = A.s[si];
  if (r < A.nrl)
    refined_corner<T, ADJ>(A, S, r);
  else
    refined_centre<T, ADJ>(A, S, r - A.nrl, si);
}

// Pairing of refined voxel v at level 0 (the level-0 kernel): u^T K9 lambda
// over its 8 corners and centre, K9 the stiffness of the refined unit voxel
// (a = 1); the host scales the sum like the structured pairing.
template <typename T, typename K>
__device__ __forceinline__ T refined_pair(const StepArgs<T>& A, int v, const T* __restrict__ hb,
                                          const T* __restrict__ chb, const T* __restrict__ lam,
                                          const T* __restrict__ clam, const K* __restrict__ k9) {
  const int uid = A.refvox_id[v];
  const int x = uid % A.un[0], y = (uid / A.un[0]) % A.un[1], z = uid / (A.un[0] * A.un[1]);
  const int i = A.fl[0] + x, j = A.fl[1] + y, k = A.fl[2] + z;
  const long long hy = A.hpx, hz = (long long)A.hpx * A.fn[1];
  const long long h0 = hidx(A, i, j, k);
  const long long l0 = lin(A, i, j, k);
  const long long ly = A.px, lz = (long long)A.px * A.ny;
  T u[9], l[9];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int a = c & 1, b = (c >> 1) & 1, d = c >> 2;
    u[c] = hb[h0 + a + b * hy + d * hz];
    l[c] = lam[l0 + a + b * ly + d * lz];
  }
  u[8] = chb[v];
  l[8] = clam[v];
  return refined_pair_sum(u, l, k9);
}

// Same-index pairing of the paper's adjoint, (u^j, lambda^j) of every unknown
// voxel (threads of the trailing blocks, per slot: the voxels, then the refined
// ones): with the step that reads lambda^j, in the slots its interior blocks
// free, instead of launches of their own that the step waited for (66 x 49 x 57,
// FEM block of half the lattice, 7.3 -> 5.1 us a level).  Large blocks keep those
// launches (the host's pairs_in_step).
template <typename T>
__device__ __noinline__ void paper_voxels(const StepArgs<T>& A, long long t) {
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2], per = nv + A.nref;
  if (t >= per * A.nslots) return;
  const int si = (int)(t / per);
  const long long r = t - per * si;
  const Slot<T>& S = A.s[si];
  double* G = A.G + (long long)si * nv;
  if (r >= nv) {
    const int v = (int)(r - nv);
    G[A.refvox_id[v]] += (double)refined_pair(A, v, S.hist_r, S.chist_r, S.cur, S.ccur, A.k9);
  } else if (!(A.refvox && A.refvox[r])) {
    const int x = (int)(r % A.un[0]);
    const long long yz = r / A.un[0];
    const int y = (int)(yz % A.un[1]), z = (int)(yz / A.un[1]);
    G[r] += (double)voxel_pair(A, S.hist_r, S.cur, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z);
  }
}

template <typename T>
__global__ void refined_pair_kernel(const __grid_constant__ StepArgs<T> A) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)A.nref * A.nslots) return;
  const int si = (int)(t / A.nref);
  const int v = (int)(t - (long long)si * A.nref);
  const Slot<T>& S = A.s[si];
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
  A.G[(long long)si * nv + A.refvox_id[v]] += (double)refined_pair(A, v, S.hist_r, S.chist_r, S.cur, S.ccur, A.k9);
}

// Damping ratio of the telegraph reading per FEM-owned node (one thread per
// node of the FEM-owned box): s_i = (tau / 2) sum_v sigma_v m_{v,i} over the
// eight voxels with a corner at i (sigma = 0 off the unknown voxels).
template <typename T>
__global__ void set_damp_kernel(const __grid_constant__ StepArgs<T> A, T* __restrict__ sd,
                                const double* __restrict__ sigma, double dt, int* flag) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
  if (t < nv) {
    const double v = sigma[t];
    if (!(v >= 0.0) || !(v <= 1e300)) atomicExch(flag, 1);
  }
  const long long nown = (long long)A.fn[0] * A.fn[1] * A.fn[2];
  if (t >= nown) return;
  const int x = (int)(t % A.fn[0]), y = (int)((t / A.fn[0]) % A.fn[1]), z = (int)(t / ((long long)A.fn[0] * A.fn[1]));
  double acc = 0.0;
  for (int c = 0; c < 8; ++c) {  // node (x, y, z) is corner c of the voxel with origin (x, y, z) - c
    const int ox = x - (c & 1), oy = y - ((c >> 1) & 1), oz = z - (c >> 2);
    if (ox < 0 || oy < 0 || oz < 0 || ox >= A.un[0] || oy >= A.un[1] || oz >= A.un[2]) continue;
    const double sv = sigma[ox + (long long)A.un[0] * (oy + (long long)A.un[1] * oz)];
    acc += sv * ((c == 0 || c == 7) ? 0.25 : 1.0 / 12.0);
  }
  sd[hidx(A, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z)] = (T)(0.5 * dt * acc);
}

template <typename T>
__global__ void set_coef_kernel(const __grid_constant__ StepArgs<T> A, T* __restrict__ W, T* __restrict__ avox,
                                const double* __restrict__ a, double a_max, int* flag) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nv = (long long)A.un[0] * A.un[1] * A.un[2];
  if (t < nv) {
    const double v = a[t];
    if (!(v <= a_max * (1.0 + 1e-12)) || !(v == v)) atomicExch(flag, 1);
    if (avox) avox[t] = (T)v;
  }
  if (t >= A.wsz) return;
  const int p[3] = {A.wx0 + (int)(t % A.wpx), A.wl[1] + (int)((t / A.wpx) % A.wn[1]),
                    A.wl[2] + (int)(t / ((long long)A.wpx * A.wn[1]))};
  const bool in_box = p[0] >= A.wl[0] && p[0] <= A.wl[0] + A.wn[0] - 1;  // else row padding
  for (int ax = 0; ax < 3; ++ax) {
    double w = 0.0;
    if (in_box && p[ax] + 1 <= A.wl[ax] + A.wn[ax] - 1) {
      const int P = ax == 0 ? 1 : 0;
      const int Q = ax == 2 ? 1 : 2;
      for (int bp = 0; bp < 2; ++bp) {
        for (int bq = 0; bq < 2; ++bq) {
          int v[3] = {p[0], p[1], p[2]};
          v[P] -= bp;
          v[Q] -= bq;
          double av = 1.0;
          if (v[0] >= A.fl[0] && v[0] < A.fl[0] + A.un[0] && v[1] >= A.fl[1] &&
              v[1] < A.fl[1] + A.un[1] && v[2] >= A.fl[2] && v[2] < A.fl[2] + A.un[2]) {
            av = a[(long long)(v[0] - A.fl[0]) +
                   (long long)A.un[0] * ((v[1] - A.fl[1]) + (long long)A.un[1] * (v[2] - A.fl[2]))];
          }
          w += av * (bp == bq ? (1.0 / 3.0) : (1.0 / 6.0));
        }
      }
    }
    W[ax * A.wsz + t] = (T)(A.ani ? w * A.kap[ax] : w);
  }
}

template <typename T>
__global__ void extract_owned_kernel(const __grid_constant__ StepArgs<T> A, const T* __restrict__ f,
                                     T* __restrict__ box) {
  const long long n = (long long)A.fn[0] * A.fn[1] * A.fn[2];
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int x = (int)(t % A.fn[0]);
  const long long r = t / A.fn[0];
  const int y = (int)(r % A.fn[1]);
  const int z = (int)(r / A.fn[1]);
  box[hidx(A, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z)] = f[lin(A, A.fl[0] + x, A.fl[1] + y, A.fl[2] + z)];
}

template <typename T>
__global__ void extract_face_kernel(const __grid_constant__ StepArgs<T> A, const T* __restrict__ f, int face,
                                    T* __restrict__ row) {
  const int ax = face >> 1;
  const int np = ax == 0 ? A.ny : A.nx, nq = ax == 2 ? A.ny : A.nz;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= np * nq) return;
  const int cp = t % np, cq = t / np;
  const int c = (face & 1) ? (ax == 0 ? A.nx : (ax == 1 ? A.ny : A.nz)) - 1 : 0;
  const int i = ax == 0 ? c : cp, j = ax == 1 ? c : (ax == 0 ? cp : cq), k = ax == 2 ? c : cq;
  row[t] = f[lin(A, i, j, k)];
}

}  // namespace

template <typename T>
void launch_extract_face(const StepArgs<T>& a, const T* field, int f, T* row, cudaStream_t st) {
  const int ax = f >> 1;
  const int n = (ax == 0 ? a.ny : a.nx) * (ax == 2 ? a.ny : a.nz);
  extract_face_kernel<T><<<(n + 255) / 256, 256, 0, st>>>(a, field, f, row);
}

template <typename T>
void launch_all_nodes(const StepArgs<T>& a, bool adjoint, cudaStream_t st) {
  const long long n = (long long)a.nx * a.ny * a.nz * a.nslots;
  if (adjoint)
    adj_all_kernel<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(a);
  else
    fwd_all_kernel<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(a);
}

template <typename T, bool ADJ>
void launch_step(const StepArgs<T>& a, bool pair, cudaStream_t st) {
  StepArgs<T> b = a;
  b.nhe = ((a.nedge + 1) / 2) * a.nslots;
  const long long nref_threads = (long long)(a.nrl + a.nref) * a.nslots;
  b.nhr = (int)((nref_threads + kStepBlock - 1) / kStepBlock);
  const long long npair = pair ? ((long long)a.un[0] * a.un[1] * a.un[2] + a.nref) * a.nslots : 0;
  const long long grid = (long long)b.nhe + b.nhr + a.nitems + (npair + kStepBlock - 1) / kStepBlock;
  // programmatic dependent launch: this level's blocks may start while the
  // previous step launch drains (they wait for it before touching its data)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kStepBlock);
  cfg.dynamicSmemBytes = kPipe<T>::bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (a.ani)
    cudaLaunchKernelEx(&cfg, step_kernel<T, ADJ, false, true>, b);
  else if (a.sdamp)
    cudaLaunchKernelEx(&cfg, step_kernel<T, ADJ, true, false>, b);
  else if (pair)
    cudaLaunchKernelEx(&cfg, step_kernel<T, false, false, false, true>, b);
  else
    cudaLaunchKernelEx(&cfg, step_kernel<T, ADJ, false, false>, b);
}

void launch_tile_step(const StepArgs<float>& a, bool adjoint, bool pair, cudaStream_t st) {
  if (adjoint) launch_step<float, true>(a, false, st);
  else launch_step<float, false>(a, pair, st);
}

template <typename T, bool ADJ>
int step_occupancy() {
  int n = 0;
  for (auto kernel : {step_kernel<T, ADJ, true, false>, step_kernel<T, ADJ, false, true>,
                      step_kernel<T, false, false, false, true>, step_kernel<T, ADJ, false, false>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPipe<T>::bytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, kStepBlock, kPipe<T>::bytes) != cudaSuccess) {
      cudaGetLastError();
      return 1;
    }
  return n > 0 ? n : 1;
}

int tile_blocks_per_sm(bool adjoint) {
  return adjoint ? step_occupancy<float, true>() : step_occupancy<float, false>();
}

template <typename T>
void launch_refined_pair(const StepArgs<T>& a, cudaStream_t st) {
  const long long n = (long long)a.nref * a.nslots;
  if (n == 0) return;
  refined_pair_kernel<T><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(a);
}

template <typename T>
void launch_pair(const StepArgs<T>& a, const T* hist, const T* lam, cudaStream_t st) {
  const long long nv = (long long)a.un[0] * a.un[1] * a.un[2];
  if (nv == 0) return;
  pair_kernel<T><<<(unsigned)((nv + 255) / 256), 256, 0, st>>>(a, hist, lam, a.G);
}

template <typename T>
void launch_set_damp(const StepArgs<T>& a, T* sdamp, const double* sigma, double dt, int* flag, cudaStream_t st) {
  const long long nv = (long long)a.un[0] * a.un[1] * a.un[2];
  const long long nown = (long long)a.fn[0] * a.fn[1] * a.fn[2];
  const long long n = nown > nv ? nown : nv;
  if (n == 0) return;
  set_damp_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, sdamp, sigma, dt, flag);
}

template <typename T>
void launch_set_coef(const StepArgs<T>& a, T* W, T* avox, const double* acoef, double a_max, int* flag,
                     cudaStream_t st) {
  const long long nv = (long long)a.un[0] * a.un[1] * a.un[2];
  const long long n = a.wsz > nv ? a.wsz : nv;
  if (n == 0) return;
  set_coef_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, W, avox, acoef, a_max, flag);
}

template <typename T>
void launch_extract_owned(const StepArgs<T>& a, const T* field, T* box, cudaStream_t st) {
  const long long n = (long long)a.fn[0] * a.fn[1] * a.fn[2];
  if (n == 0) return;
  extract_owned_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, field, box);
}

#define HYB_INSTANTIATE(T)                                                                       \
  template void launch_all_nodes<T>(const StepArgs<T>&, bool, cudaStream_t);                     \
  template void launch_pair<T>(const StepArgs<T>&, const T*, const T*, cudaStream_t);            \
  template void launch_set_coef<T>(const StepArgs<T>&, T*, T*, const double*, double, int*,     \
                                   cudaStream_t);                                                \
  template void launch_set_damp<T>(const StepArgs<T>&, T*, const double*, double, int*, cudaStream_t); \
  template void launch_extract_owned<T>(const StepArgs<T>&, const T*, T*, cudaStream_t);              \
  template void launch_extract_face<T>(const StepArgs<T>&, const T*, int, T*, cudaStream_t);        \
  template void launch_refined_pair<T>(const StepArgs<T>&, cudaStream_t);

HYB_INSTANTIATE(float)
HYB_INSTANTIATE(double)

}  // namespace hyb
