// The sweep kernel: a run of consecutive time levels of every slot in one
// launch, for FP64 fields (FP32 fields take the staged tiles of
// step_kernels.cu).
//
// Blocks claim work items (level, slot, item) in order and an item waits only
// for the previous level's items around it.  Items are runs of interior rows
// (16-byte groups of nodes along x, marched along z in registers), the nodes
// next to one outer face, the edge tiles (nodes within one node of two faces)
// and the rows of the refined region.  All items of a level read levels k and
// k-1 and write disjoint nodes of level k+1.
#include "async_copy.cuh"
#include "rows.cuh"

namespace hyb {
namespace {

// ---- the sweep kernel: consecutive levels of every slot in one launch ----
// Work items of one level of one slot: blocks of quads of the interior, nodes
// next to one outer face, edge tiles, rows of the refined region.
enum ItemKind { kInterior = 0, kFace = 1, kEdgeZ = 2, kEdgeXY = 3, kRefined = 4 };

// The "edge set": every node whose coordinate is near a face (0, 1, n-2 or
// n-1) on at least two axes.  It is cut into tiles of 128 threads: along z 4 x 4
// near coordinates x 8 positions (bar = 2), along y and x at one z end 4 near
// coordinates x 2 planes x 16 positions (bar = 1, 0), and the 4 x 4 x 2 corner
// nodes of one z end (bar = -1).  Within a tile every absorbing coupling stays
// inside the tile.  Returns false for idle threads; q[] holds the near index
// (0..3 -> 0, 1, n-2, n-1) per axis (-1: mid) and nf the number of axes on
// which the node is on a face.
struct EdgeTile {
  int bar;         // -2: no tile
  int end;         // z end of the bars along x and y and of the corners (0: low, 1: high)
  int pos0, pos1;  // node range along the bar
};

template <typename T>
__device__ __forceinline__ bool edge_tile_node(const SweepArgs<T>& A, const EdgeTile& E, int t, int& i, int& j, int& k,
                                               int q[3], int& nf) {
  const int nx = A.nx, ny = A.ny, nz = A.nz;
  auto nr = [](int qq, int n) { return qq < 2 ? qq : n - 4 + qq; };
  if (E.bar == -2) return false;
  const int lo = t & 3, hi = (t >> 2) & 3;
  int pos = 0;
  if (E.bar < 0) {
    if (t >= 32) return false;
    q[0] = lo;
    q[1] = hi;
    q[2] = 2 * E.end + (t >> 4);
  } else if (E.bar == 2) {
    pos = E.pos0 + (t >> 4);
    if (pos >= E.pos1) return false;
    q[0] = lo;
    q[1] = hi;
    q[2] = -1;
  } else {
    pos = E.pos0 + (t >> 3);
    if (pos >= E.pos1) return false;
    q[0] = E.bar == 0 ? -1 : lo;
    q[1] = E.bar == 1 ? -1 : lo;
    q[2] = 2 * E.end + ((t >> 2) & 1);
  }
  i = q[0] < 0 ? pos : nr(q[0], nx);
  j = q[1] < 0 ? pos : nr(q[1], ny);
  k = q[2] < 0 ? pos : nr(q[2], nz);
  nf = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) nf += (q[a] == 0 || q[a] == 3) ? 1 : 0;
  return true;
}

// Thread index, inside the same tile, of the node with near index qn on
// axis ax (the other coordinates unchanged; on z the same end).
__device__ __forceinline__ int edge_tile_peer(int t, int bar, int ax, int qn) {
  if (ax == 2) {  // (not on bars along z)
    const int sh = bar < 0 ? 4 : 2;
    return (t & ~(1 << sh)) | ((qn & 1) << sh);
  }
  const int sh = (bar < 0 || bar == 2) ? 2 * ax : 0;
  return (t & ~(3 << sh)) | (qn << sh);
}

// Barrier of the block's row threads (all but the producer warp).
__device__ __forceinline__ void row_sync() {
  asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x - kServiceThreads) : "memory");
}

// Edge tile of the forward step.  Levels by the number of faces a node lies
// on: nodes on no face take their interior row, then face, edge and corner
// nodes; an absorbing row (Eq. (eq:abs2)) reads the new values of its
// inward neighbours, one level down in the same tile, from shared memory.
// Every row thread of the block calls it (it synchronises); nv holds 128 values.
template <typename T, bool ANI>
__device__ __forceinline__ void fwd_edge_tile(const SweepArgs<T>& A, const Slot<T>& S, const EdgeTile& E, int t, T* nv) {
  int i = 0, j = 0, k = 0, nf = -1, q[3];
  const bool valid = edge_tile_node(A, E, t, i, j, k, q, nf);
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
  row_sync();
  for (int level = 1; level <= 3; ++level) {
    T v = T(0);
    const bool mine = valid && fb && __popc(fall) == level;
    if (mine) {
      T acc = T(0);
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const int fa = (fb >> (2 * ax)) & 3;
        if (!fa) continue;
        const int t1 = edge_tile_peer(t, E.bar, ax, (fa & 1) ? 1 : 2);
        acc += cin[ax] - (ANI ? A.ra[ax] : A.r) * nv[t1];
      }
      v = (ANI ? abc_self(A, fb) : A.r) * cself + over_faces(acc, __popc(fb));
    }
    row_sync();
    if (mine) nv[t] = v;
    row_sync();
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
__device__ __forceinline__ void adj_edge_tile(const SweepArgs<T>& A, const Slot<T>& S, const EdgeTile& E, int t, T* lam) {
  int i = 0, j = 0, k = 0, nf = -1, q[3];
  const bool valid = edge_tile_node(A, E, t, i, j, k, q, nf);
  lam[t] = valid ? adj_rhs_inl<T, ANI>(A, S, i, j, k) : T(0);
  row_sync();
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
        v -= over_faces(ANI ? A.ra[ax] : A.r, __popc(fbb)) * lam[edge_tile_peer(t, E.bar, ax, q[ax] == 1 ? 0 : 3)];
      }
    }
    row_sync();
    if (mine) lam[t] = v;
    row_sync();
  }
  if (valid) S.next[lin(A, i, j, k)] = lam[t];
}

// 16-byte groups of consecutive nodes along x ("quads"; rows start on 32-byte
// boundaries, so quads are aligned).
template <typename T>
struct Quad {
  static constexpr int V = 16 / (int)sizeof(T);
};
__device__ __forceinline__ void ldq(double (&v)[2], const double* p) {
  const double2 f = *reinterpret_cast<const double2*>(p);
  v[0] = f.x, v[1] = f.y;
}
__device__ __forceinline__ void stq(double* p, const double (&v)[2]) {
  *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}

// Unit-weight lattice rows (FP64) from differences: the z differences are carried from plane to
// plane and the x differences shared between neighbouring nodes, which takes
// 12.5 operations a node where the six differences of each node take 14 (the
// FP64 pipe bounds these rows: 2 lanes per SM and clock).
__device__ __forceinline__ void lattice_rows(double (&val)[2], const double (&c)[2], const double (&dx)[3],
                                             const double (&dym)[2], const double (&dyp)[2], const double (&dzm)[2],
                                             const double (&dzp)[2], const double (&pv)[2], double c2) {
#pragma unroll
  for (int e = 0; e < 2; ++e)
    val[e] = c[e] + ((c[e] - pv[e]) + c2 * (((dx[e + 1] - dx[e]) + (dyp[e] - dym[e])) + (dzp[e] - dzm[e])));
}

// One row with per-axis weights kap: the forward row, or the transposed row
// in the gathered order of adj_rhs.
template <typename T, bool ADJ>
__device__ __forceinline__ T ani_row(const SweepArgs<T>& A, T c, T xm, T xp, T ym, T yp, T zm, T zp, T pv) {
  if constexpr (ADJ) {
    const T cx = A.c2 * A.kapt[0], cy = A.c2 * A.kapt[1], cz = A.c2 * A.kapt[2];
    T rhs = (T(2) + A.c2 * A.kdiag) * c;
    rhs += cx * xm;
    rhs += cx * xp;
    rhs += cy * ym;
    rhs += cy * yp;
    rhs += cz * zm;
    rhs += cz * zp;
    return rhs - pv;
  } else {
    const T lx = (xm - c) + (xp - c), ly = (ym - c) + (yp - c), lz = (zm - c) + (zp - c);
    return c + ((c - pv) + A.c2 * ((A.kapt[0] * lx + A.kapt[1] * ly) + A.kapt[2] * lz));
  }
}

// A row with edge weights (FEM-owned node) from the differences u_nb - u^k.
template <typename T, bool TEL>
__device__ __forceinline__ T fem_diff_row(T c, T dxm, T dxp, T dym, T dyp, T dzm, T dzp, T pv, T wxm, T wxp, T wym,
                                          T wyp, T wzm, T wzp, T sd, T c2) {
  const T lap = wxp * dxp + wxm * dxm + wyp * dyp + wym * dym + wzp * dzp + wzm * dzm;
  if constexpr (TEL) return c + ((c - pv) * (T(1) - sd) + c2 * lap) / (T(1) + sd);
  return c + ((c - pv) + c2 * lap);
}

// The same from the values: forward, damped (telegraph, sd the node's damping
// ratio), or with per-axis steps transposed.
template <typename T, bool ADJ, bool TEL, bool ANI>
__device__ __forceinline__ T fem_row(const SweepArgs<T>& A, T c, T xm, T xp, T ym, T yp, T zm, T zp, T pv, T wxm, T wxp,
                                     T wym, T wyp, T wzm, T wzp, T sd) {
  if constexpr (ADJ && ANI) {
    T rhs = (T(2) + A.c2 * -(wxp + wxm + wyp + wym + wzp + wzm)) * c;
    rhs += A.c2 * wxm * xm;
    rhs += A.c2 * wxp * xp;
    rhs += A.c2 * wym * ym;
    rhs += A.c2 * wyp * yp;
    rhs += A.c2 * wzm * zm;
    rhs += A.c2 * wzp * zp;
    return rhs - pv;
  }
  return fem_diff_row<T, TEL>(c, xm - c, xp - c, ym - c, yp - c, zm - c, zp - c, pv, wxm, wxp, wym, wyp, wzm, wzp, sd,
                              A.c2);
}

// Faces whose rows the interior items take along: absorbing in this step (and,
// transposed, in the next one: then nothing but values at hand enters).  The
// other faces' nodes and their neighbours are left to the face items, the x
// faces among them, whose few lanes would cost every warp of a row a pass of
// the FP64 pipe.
template <typename T, StepMode M>
__device__ __forceinline__ int inline_faces(const Slot<T>& S) {
  const int f = M == kAdjoint ? (S.mask_f & S.mask_c) : (M == kForward ? S.mask_f : 0);
  return f & ~3;
}

// Stage and phase of the ring position a side of the pipeline is at.
struct RingPos {
  int st;
  unsigned ph;
  __device__ __forceinline__ void next(int ns) {
    if (++st == ns) {
      st = 0;
      ph ^= 1u;
    }
  }
};

// Barriers of a block's pipelines.
struct Bars {
  uint64_t full[kMaxStages], empty[kMaxStages];  // stages: landed / released by every row warp
  uint64_t qfull[2], qempty[2];                  // items: published / done
};

// Interior rows (nodes 1 .. n-2 on every axis; the edge set and the nodes next
// to a face that is not inline are left out).  An item is up to one quad per row
// thread, consecutive quads of the rows of one plane, one per row thread whatever the
// lattice's width (so every warp is full), marched through the slab's planes.
// The producer warp copies each plane's run of memory that holds the item's
// rows and the rows above and below them (u^k, and the item's rows of u^{k-1})
// into a ring of shared-memory stages with bulk copies, ahead of the march and
// into the next item.  u^k of the planes below and above stays in registers;
// the x neighbours come from the neighbouring lanes.
template <typename T>
struct InteriorRun {  // the part both sides compute
  int za, zb;         // planes
  int first, n;       // quads of the plane: first, count
  long long a0, a1;   // memory range of the item's quads within a plane (nodes)
  __device__ __forceinline__ InteriorRun(const SweepArgs<T>& A, int slab, int first_quad) {
    constexpr int V = 16 / (int)sizeof(T);
    za = 1 + slab * A.slabz;
    zb = min(za + A.slabz, A.nz - 1);
    first = first_quad;
    n = min((int)blockDim.x - kServiceThreads, (A.ny - 2) * A.nqx - first);
    const int j0 = first / A.nqx, j1 = (first + n - 1) / A.nqx;
    a0 = (long long)A.px * (1 + j0) + V * (first - j0 * A.nqx);
    a1 = (long long)A.px * (1 + j1) + V * (first + n - 1 - j1 * A.nqx) + V;
  }
};

// Producer side of an interior item (one thread): plane stages za - 1 (the
// item's rows only), za .. zb - 1 (with the rows around, one quad further for
// the pairing, and u^{k-1}), zb (with the rows around).  False when a wait ran out (no copy is issued after that).
template <typename T>
__device__ __forceinline__ bool interior_produce(const SweepArgs<T>& A, Bars* B, T* ring, RingPos& rp, const T* cur,
                                                 const T* prev, int slab, int first, long long budget, unsigned& issued) {
  const InteriorRun<T> R(A, slab, first);
  const long long pl = (long long)A.px * A.ny;
  const uint32_t run = (uint32_t)((R.a1 - R.a0) * sizeof(T));
  constexpr int V = 16 / (int)sizeof(T);
  for (int k = R.za - 1; k <= R.zb; ++k) {
    if (!mbar_wait_idle(B->empty + rp.st, rp.ph ^ 1u, budget, A.err)) return false;
    fence_proxy_async_shared();  // (the row threads' reads of the stage before the copies into it)
    T* c = ring + (size_t)rp.st * A.nstage;
    uint64_t* bar = B->full + rp.st;
    const T* src = cur + pl * k + R.a0;
    const bool halo = k >= R.za, pv = halo && k < R.zb;
    if (!halo) {
      mbar_arrive_expect_tx(bar, run);
      bulk_load(c + A.ccen, src, run, bar);
    } else if (!A.split) {
      const uint32_t all = run + (uint32_t)((2 * A.px + V) * sizeof(T));
      mbar_arrive_expect_tx(bar, all + (pv ? run : 0u));
      bulk_load(c, src - A.px, all, bar);
    } else {
      mbar_arrive_expect_tx(bar, 3 * run + 3 * (uint32_t)(V * sizeof(T)) + (pv ? run : 0u));
      bulk_load(c + A.ccen - A.yo, src - A.px, run, bar);
      bulk_load(c + A.ccen - V, src - V, run + 2 * (uint32_t)(V * sizeof(T)), bar);
      bulk_load(c + A.ccen + A.yo, src + A.px, run + (uint32_t)(V * sizeof(T)), bar);
    }
    if (pv) bulk_load(c + A.ncur, prev + pl * k + R.a0, run, bar);
    rp.next(A.ns);
    ++issued;
  }
  return true;
}

// The face node b next to the node m (value cm, new value v, coefficient coef
// of m's row on b) across an inline face f: forward Eq. (eq:abs2); transposed
// b's row, and m's corrected for it.
template <typename T, bool ADJ>
__device__ __forceinline__ T inline_face(const Slot<T>& S, T rf, T c2, int f, T ub, T cm, T& v, T coef, T obs) {
  if constexpr (!ADJ) return rf * ub + (cm - rf * v);
  T lb = rf * ub;
  lb += c2 * coef * cm;
  lb += obs;
  v += ub - c2 * coef * ub;
  if ((S.mask_e >> f) & 1) v -= rf * lb;
  return lb;
}

// The rows of one warp through an interior item's planes.  FEM: the warp has
// FEM-owned nodes in the item (edge weights, history, pairing); the other
// warps run the short loop.  Every lane computes all of its quad's nodes and
// stores those that are the item's.
template <typename T, StepMode M, bool TEL, bool ANI, bool FEM>
__device__ __forceinline__ void interior_march(const SweepArgs<T>& A, const Slot<T>& S, Bars* B, const T* ring,
                                               RingPos& rp, int si, const InteriorRun<T>& R) {
  constexpr int V = Quad<T>::V;
  constexpr bool ADJ = M == kAdjoint, PAIR = FEM && M != kForward;
  constexpr bool DIF = !ANI;  // rows from differences: zm carries u - (u below)
  constexpr unsigned kAll = (1u << V) - 1;
  const bool valid = (int)threadIdx.x < R.n;
  const int t = R.first + (valid ? (int)threadIdx.x : R.n - 1);
  const int jr = t / A.nqx, qx = t - jr * A.nqx;
  const int j = 1 + jr, i0 = V * qx;
  const int lane = (int)threadIdx.x & 31;
  const int px = A.px, yo = A.yo, nstage = A.nstage, ns = A.ns;
  const long long pl = (long long)px * A.ny;
  const int inl = inline_faces<T, M>(S);
  // elements: off the x faces' neighbours, FEM-owned
  unsigned mid = 0, fem = 0;
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int i = i0 + e;
    if (i >= 2 && i <= A.nx - 3) mid |= 1u << e;
    if (FEM && i >= A.fl[0] && i <= A.fh[0] && j >= A.fl[1] && j <= A.fh[1]) fem |= 1u << e;
  }
  const int fy = j == 1 ? 2 : (j == A.ny - 2 ? 3 : -1);  // the y face next to the row
  if (!valid) mid = 0;
  const bool anyfy = __any_sync(0xffffffffu, fy >= 0);
  // elements written on the planes off the z faces
  const unsigned wr0 = fy < 0 || ((inl >> fy) & 1) ? mid : 0;
  const int so = (int)(i0 + (long long)px * j - R.a0);  // this quad in the item's run
  const T* const base = ring + A.ccen + so;
  const int pvo = A.ncur - A.ccen;
  const T c2 = A.c2;
  T* o = S.next + (i0 + (long long)px * j + pl * R.za);
  const int last = A.fl[0] + A.un[0] - 1;  // x of the last voxel origin
  const bool over = PAIR && i0 + V - 1 <= last;
  auto wait = [&](const RingPos& q) {
    if (!mbar_try(B->full + q.st, q.ph) && !mbar_wait_slow(B->full + q.st, q.ph, A.wait, A.err)) atomicExch(A.err, 1);
  };
  auto release = [&](const RingPos& q) {
    __syncwarp();  // (the warp's reads of the stage are done)
    if (lane == 0) mbar_arrive(B->empty + q.st);
  };
  T zm[V], c[V], zp[V], pv[V];
  wait(rp);
  ldq(zm, base + rp.st * nstage);
  release(rp);
  rp.next(ns);
  wait(rp);
  const T* C = base + rp.st * nstage;
  ldq(c, C);
  if constexpr (DIF) {
#pragma unroll
    for (int e = 0; e < V; ++e) zm[e] = c[e] - zm[e];
  }
  for (int k = R.za; k < R.zb; ++k, o += pl) {
    RingPos up = rp;
    up.next(ns);
    const T* U = base + up.st * nstage;
    const int fz = k == 1 ? 4 : (k == A.nz - 2 ? 5 : -1);  // (uniform)
    unsigned wr = wr0;  // elements this thread writes
    if (fz >= 0) wr = fy < 0 && ((inl >> fz) & 1) ? mid : 0;
    const unsigned fm = FEM && k >= A.fl[2] && k <= A.fh[2] ? fem & wr : 0;
    T wl = T(0), wx[V], wy0[V], wy1[V], wz0[V], wz1[V], sd[V];
    T h00[V], h10[V], h01[V], h11[V], a00 = T(0), a10 = T(0), a01 = T(0), a11 = T(0);
    unsigned rf = 0;  // refinement flags, one byte per element
    long long h = 0;
    bool pairq = false;
    if constexpr (FEM) {
      if (fm) {  // (global loads: before the wait below)
        const long long w = widx(A, i0, j, k), wz = (long long)A.wpx * A.wn[1];
        const T* W = S.W + w;
        if (fm & 1) wl = W[-1];
        ldq(wx, W);
        ldq(wy1, W + A.wsz);
        ldq(wy0, W + A.wsz - A.wpx);
        ldq(wz1, W + 2 * A.wsz);
        ldq(wz0, W + 2 * A.wsz - wz);
        h = hidx(A, i0, j, k);
        if constexpr (TEL) ldq(sd, A.sdamp + h);
        if (A.nref) rf = *reinterpret_cast<const unsigned short*>(A.rmask + h);
        if constexpr (PAIR) {
          pairq = S.hist_r && j - A.fl[1] < A.un[1] && k - A.fl[2] < A.un[2];
          if (pairq) {
            // voxels with their origin at the quad's nodes: u and lambda on rows
            // j, j + 1 of planes k, k + 1, one node beyond the quad
            const long long hy = A.hpx, hz = (long long)A.hpx * A.fn[1];
            const T* H = S.hist_r + h;
            ldq(h00, H);
            ldq(h10, H + hy);
            ldq(h01, H + hz);
            ldq(h11, H + hz + hy);
            if (over) {
              a00 = H[V];
              a10 = H[hy + V];
              a01 = H[hz + V];
              a11 = H[hz + hy + V];
            }
          }
        }
      }
    }
    T ym[V], yp[V];
    ldq(ym, C - yo);
    ldq(yp, C + yo);
    ldq(pv, C + pvo);
    const T xl = C[-1], xr = C[V];
    const T b10 = PAIR ? C[yo + V] : T(0);
    wait(up);
    ldq(zp, U);
    release(rp);
    T val[V];
    if constexpr (DIF) {
      T dx[V + 1], dym[V], dyp[V], dzp[V];
#pragma unroll
      for (int e = 0; e <= V; ++e) dx[e] = (e < V ? c[e] : xr) - (e ? c[e - 1] : xl);
#pragma unroll
      for (int e = 0; e < V; ++e) {
        dym[e] = c[e] - ym[e];
        dyp[e] = yp[e] - c[e];
        dzp[e] = zp[e] - c[e];
      }
      lattice_rows(val, c, dx, dym, dyp, zm, dzp, pv, c2);
      if (FEM && fm) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const T v = fem_diff_row<T, TEL>(c[e], -dx[e], dx[e + 1], -dym[e], dyp[e], -zm[e], dzp[e], pv[e],
                                           e ? wx[e - 1] : wl, wx[e], wy0[e], wy1[e], wz0[e], wz1[e],
                                           TEL ? sd[e] : T(0), c2);
          val[e] = (fm >> e) & 1 ? v : val[e];
        }
      }
#pragma unroll
      for (int e = 0; e < V; ++e) zm[e] = dzp[e];
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e)
        val[e] = ani_row<T, ADJ>(A, c[e], e ? c[e - 1] : xl, e < V - 1 ? c[e + 1] : xr, ym[e], yp[e], zm[e], zp[e],
                                 pv[e]);
      if (FEM && fm) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const T v = fem_row<T, ADJ, TEL, ANI>(A, c[e], e ? c[e - 1] : xl, e < V - 1 ? c[e + 1] : xr, ym[e], yp[e],
                                                zm[e], zp[e], pv[e], e ? wx[e - 1] : wl, wx[e], wy0[e], wy1[e],
                                                wz0[e], wz1[e], TEL ? sd[e] : T(0));
          val[e] = (fm >> e) & 1 ? v : val[e];
        }
      }
#pragma unroll
      for (int e = 0; e < V; ++e) zm[e] = c[e];
    }
    if constexpr (FEM) {
      if (fm) {
        unsigned hw = fm;  // FEM-owned elements the refined rows do not write
#pragma unroll
        for (int e = 0; e < V; ++e)
          if ((rf >> (8 * e)) & 1) hw &= ~(1u << e);
        wr &= hw | ~fm;
        if constexpr (M == kForward) {
          if (S.hist_w) {
            T hv[V];
#pragma unroll
            for (int e = 0; e < V; ++e) hv[e] = TEL ? val[e] - pv[e] : val[e];
            if (hw == kAll) {
              stq(S.hist_w + h, hv);
            } else {
#pragma unroll
              for (int e = 0; e < V; ++e)
                if ((hw >> e) & 1) S.hist_w[h + e] = hv[e];
            }
          }
        }
        if constexpr (PAIR) {
          if (pairq) {
            const int vj = j - A.fl[1], vk = k - A.fl[2];
            T q[V];
            ldq(q, U + yo);
            const T b01 = over ? U[V] : T(0), b11 = over ? U[yo + V] : T(0);
            double* G = A.G + ((long long)si * A.un[2] + vk) * ((long long)A.un[0] * A.un[1]) +
                        (long long)A.un[0] * vj + (i0 - A.fl[0]);
#pragma unroll
            for (int e = 0; e < V; ++e) {
              if (!((fm >> e) & 1) || i0 + e > last || ((rf >> (8 * e)) & 2)) continue;
              const bool in = e < V - 1;
              const int f = in ? e + 1 : e;
              const T uu[8] = {h00[e], in ? h00[f] : a00, h10[e], in ? h10[f] : a10,
                               h01[e], in ? h01[f] : a01, h11[e], in ? h11[f] : a11};
              const T ll[8] = {c[e],  in ? c[f] : xr,   yp[e], in ? yp[f] : b10,
                               zp[e], in ? zp[f] : b01, q[e],  in ? q[f] : b11};
              atomicAdd(G + e, (double)(TEL ? damp_sum(uu, ll) : (ANI ? pair_sum_ani(A, uu, ll) : pair_sum(uu, ll))));
            }
          }
        }
      }
    }
    if (anyfy || fz >= 0) {  // (warp-uniform) rows next to a y face, the plane next to a z face
      if ((fy >= 0 || fz >= 0) && wr) {
        const int f = fy >= 0 ? fy : fz;
        T ub[V];
        if (fy >= 0) {
#pragma unroll
          for (int e = 0; e < V; ++e) ub[e] = fy == 2 ? ym[e] : yp[e];
        } else if (fz == 5) {
#pragma unroll
          for (int e = 0; e < V; ++e) ub[e] = zp[e];
        } else {
          ldq(ub, S.cur + (o - S.next) - pl);
        }
        T* ob = o + (fy >= 0 ? (fy == 2 ? -px : px) : (fz == 4 ? -pl : pl));
        const bool obs = S.obs_face == f;
        const int idx = i0 + A.nx * (fy >= 0 ? k : j);
#pragma unroll
        for (int e = 0; e < V; ++e) {
          if (!((wr >> e) & 1)) continue;
          T coef = ANI ? A.kapt[f >> 1] : T(1);
          if (FEM && ADJ && ((fm >> e) & 1)) coef = f == 2 ? wy0[e] : (f == 3 ? wy1[e] : (f == 4 ? wz0[e] : wz1[e]));
          const T vb = inline_face<T, ADJ>(S, ANI ? A.ra[f >> 1] : A.r, c2, f, ub[e], c[e], val[e], coef,
                                           ADJ && obs && S.obs_r ? S.obs_r[idx + e] : T(0));
          ob[e] = vb;
          if (!ADJ && obs && S.obs_w) S.obs_w[idx + e] = vb;
        }
      }
    }
    if (wr == kAll) {
      stq(o, val);
    } else if (wr) {
#pragma unroll
      for (int e = 0; e < V; ++e)
        if ((wr >> e) & 1) o[e] = val[e];
    }
#pragma unroll
    for (int e = 0; e < V; ++e) c[e] = zp[e];
    rp = up;
    C = U;
  }
  release(rp);
  rp.next(ns);
}

template <typename T, StepMode M, bool TEL, bool ANI>
__device__ __forceinline__ void interior_item(const SweepArgs<T>& A, const Slot<T>& S, Bars* B, const T* ring,
                                              RingPos& rp, int si, int slab, int first) {
  const InteriorRun<T> R(A, slab, first);
  // rows of the warp's quads against the FEM block's (an x test would seldom help)
  const int w0 = R.first + ((int)threadIdx.x & ~31), w1 = min(w0 + 31, R.first + R.n - 1);
  const bool fem = w0 <= w1 && A.fl[0] <= A.fh[0] && 1 + w0 / A.nqx <= A.fh[1] && 1 + w1 / A.nqx >= A.fl[1] &&
                   R.za <= A.fh[2] && R.zb > A.fl[2];
  if (fem) interior_march<T, M, TEL, ANI, true>(A, S, B, ring, rp, si, R);
  else interior_march<T, M, false, ANI, false>(A, S, B, ring, rp, si, R);
}

// The node m = (i, j, k) one step inside exactly one outer face that is not
// inline (axis ax, side sd = -1 / +1) and the face node b next to it.
// Forward: m's row, then the absorbing row of Eq. (eq:abs2) at b from u^k at b
// and m and the new value at m, or b's mirror-ghost row with the source flux.
// Transposed: b's row in closed form (no transposed absorbing coupling
// reaches it), from lambda^{j+1} at b and m, the coefficient of m's row on b
// and lambda^{j+2} at b; then m's row, corrected for b's coupling.
template <typename T, StepMode M, bool ANI>
__device__ __forceinline__ void face_pair(const SweepArgs<T>& A, const Slot<T>& S, int si, int i, int j, int k, int ax,
                                          int sd) {
  constexpr bool ADJ = M == kAdjoint;
  const T* u = S.cur;
  const long long id = lin(A, i, j, k);
  const long long sy = A.px, sz = (long long)A.px * A.ny;
  const long long st = sd * (ax == 0 ? 1LL : (ax == 1 ? sy : sz));
  const long long o1 = ax == 0 ? sy : 1, o2 = ax == 2 ? sy : sz;  // in-face axes
  const long long b = id + st;
  const int f = 2 * ax + (sd > 0 ? 1 : 0);
  if ((inline_faces<T, M>(S) >> f) & 1) return;  // (the interior items take it along)
  const bool abc = (S.mask_f >> f) & 1;
  const T c0 = u[id], xm = u[id - 1], xp = u[id + 1], ym = u[id - sy], yp = u[id + sy], zm = u[id - sz], zp = u[id + sz];
  const T pv = S.prev[id];
  const T ub = u[b], pb = S.prev[b];
  T n1m = T(0), n1p = T(0), n2m = T(0), n2p = T(0);
  if (!abc) {
    n1m = u[b - o1];
    n1p = u[b + o1];
    n2m = u[b - o2];
    n2p = u[b + o2];
  }
  const T rf = ANI ? A.ra[ax] : A.r;
  const T kax = ANI ? A.kapt[ax] : T(1), k1 = ANI ? A.kapt[ax == 0 ? 1 : 0] : T(1), k2 = ANI ? A.kapt[ax == 2 ? 1 : 2] : T(1);
  const bool fo = fem_owned(A, i, j, k);
  T val, coef_mb = kax;  // m's row; its coefficient on b
  if (fo) {
    const long long w = widx(A, i, j, k), wy = A.wpx, wz = (long long)A.wpx * A.wn[1];
    const T* W = S.W + w;
    const T wxp = W[0], wxm = W[-1], wyp = W[A.wsz], wym = W[A.wsz - wy], wzp = W[2 * A.wsz], wzm = W[2 * A.wsz - wz];
    coef_mb = ax == 0 ? (sd > 0 ? wxp : wxm) : (ax == 1 ? (sd > 0 ? wyp : wym) : (sd > 0 ? wzp : wzm));
    val = fem_row<T, ADJ, false, ANI>(A, c0, xm, xp, ym, yp, zm, zp, pv, wxm, wxp, wym, wyp, wzm, wzp, T(0));
  } else if constexpr (ANI) {
    val = ani_row<T, ADJ>(A, c0, xm, xp, ym, yp, zm, zp, pv);
  } else {
    const T lap = (((xp - c0) - (c0 - xm)) + ((yp - c0) - (c0 - ym))) + ((zp - c0) - (c0 - zm));
    val = c0 + ((c0 - pv) + A.c2 * lap);
  }
  const int bi = i + (ax == 0 ? sd : 0), bj = j + (ax == 1 ? sd : 0), bk = k + (ax == 2 ? sd : 0);
  const int fi = face_index(f, bi, bj, bk, A.nx, A.ny);
  if constexpr (!ADJ) {
    T vb;
    if (abc) {
      vb = rf * ub + (c0 - rf * val);
    } else {
      T lb = kax * (T(2) * (c0 - ub));
      lb += k1 * ((n1m - ub) + (n1p - ub));
      lb += k2 * ((n2m - ub) + (n2p - ub));
      vb = ub + ((ub - pb) + A.c2 * lb);
      if ((S.src_mask >> f) & 1) vb += src_term(S, f, bi, bj, bk);
      if (S.inj && S.obs_face == f) vb += S.inj_scale * T(2) * S.inj[fi];
    }
    S.next[b] = vb;
    if (S.obs_w && S.obs_face == f) S.obs_w[fi] = vb;
    if (fo && S.hist_w) S.hist_w[hidx(A, i, j, k)] = val;
  } else {
    T lb = abc ? rf * ub : (T(2) + A.c2 * (ANI ? A.kdiag : T(-6))) * ub;
    lb += A.c2 * coef_mb * c0;
    if (!abc) {
      lb += A.c2 * k1 * (n1m + n1p);
      lb += A.c2 * k2 * (n2m + n2p);
    }
    if (!((S.mask_c >> f) & 1)) lb -= pb;
    if (S.obs_r && S.obs_face == f) lb += S.obs_r[fi];
    val += (abc ? ub : T(2) * A.c2 * kax * ub) - A.c2 * coef_mb * ub;
    if ((S.mask_e >> f) & 1) val -= rf * lb;
    S.next[b] = lb;
  }
  S.next[id] = val;
  if constexpr (M != kForward) pair_if_voxel<T, ANI>(A, S, si, i, j, k);
}

// One entry of a slab's list of nodes one step inside exactly one face, in
// the order z faces (first and last slab), y faces, x faces.
template <typename T, StepMode M, bool ANI>
__device__ __forceinline__ void face_entry(const SweepArgs<T>& A, const Slot<T>& S, int si, int slab, unsigned t) {
  const unsigned mx = A.nx - 4, my = A.ny - 4;
  const int k0 = max(1 + slab * A.slabz, 2), k1 = min(1 + (slab + 1) * A.slabz, A.nz - 2);
  const unsigned mz = max(k1 - k0, 0);
  const unsigned nlo = slab == 0 ? mx * my : 0, nhi = slab == A.nslab - 1 ? mx * my : 0;
  if (t < nlo + nhi) {
    const bool hi = t >= nlo;
    if (hi) t -= nlo;
    const int y = t / mx, x = t - y * mx;
    face_pair<T, M, ANI>(A, S, si, 2 + x, 2 + y, hi ? A.nz - 2 : 1, 2, hi ? 1 : -1);
    return;
  }
  t -= nlo + nhi;
  if (t < 2 * mx * mz) {
    const bool hi = t >= mx * mz;
    if (hi) t -= mx * mz;
    const int z = t / mx, x = t - z * mx;
    face_pair<T, M, ANI>(A, S, si, 2 + x, hi ? A.ny - 2 : 1, k0 + z, 1, hi ? 1 : -1);
    return;
  }
  t -= 2 * mx * mz;
  if (t < 2 * my * mz) {
    const bool hi = t >= my * mz;
    if (hi) t -= my * mz;
    const int z = t / my, y = t - z * my;
    face_pair<T, M, ANI>(A, S, si, hi ? A.nx - 2 : 1, 2 + y, k0 + z, 0, hi ? 1 : -1);
  }
}

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

// Absorbing faces of the step leaving t_k = k dt, and the faces carrying the
// flux (an entry face carries it while t_k <= its switch time).
template <typename T>
__device__ __forceinline__ int phase(const SweepArgs<T>& A, int si, int k, int* flux) {
  const double t = __dmul_rn((double)k, A.dt);
  int sm = 0;
#pragma unroll
  for (int f = 0; f < 6; ++f)
    if (((A.entry[si] >> f) & 1) && t <= A.tsw[si][f]) sm |= 1 << f;
  if (flux) *flux = sm;
  return A.abc_mask & ~sm;
}

// Ring slot of `cur`, `prev` (which 1, 2) at level l of the launch.
template <typename T>
__device__ __forceinline__ int ring_slot(const SweepArgs<T>& A, int l, int which) {
  const int r = (A.ring0 + A.dir * (l % 3) + 3) % 3;
  if (which == 0) return r;
  return (r + (which == 1 ? 3 - A.dir : 3 + A.dir)) % 3;
}

template <typename T>
__device__ __forceinline__ T* ring_field(const SweepArgs<T>& A, int r, int si) {
  return A.fbase + ((long long)r * A.nslots + si) * A.Np;
}

// Every slot at every level of a launch (A.table), from the slots of its first level.
template <typename T, StepMode M>
__global__ void slots_kernel(const __grid_constant__ SweepArgs<T> A) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= A.nlev * A.nslots) return;
  const int l = q / A.nslots, si = q - l * A.nslots;
  Slot<T>* S = A.table + q;
  *S = A.s[si];
  const int step = A.k0 + A.dir * l;
  const int r = ring_slot(A, l, 0), rp = ring_slot(A, l, 1), rn = ring_slot(A, l, 2);
  S->cur = ring_field(A, r, si);
  S->prev = ring_field(A, rp, si);
  S->next = ring_field(A, rn, si);
  if (A.nref) {
    S->ccur = A.cbase + ((long long)r * A.nslots + si) * A.nref;
    S->cprev = A.cbase + ((long long)rp * A.nslots + si) * A.nref;
    S->cnext = A.cbase + ((long long)rn * A.nslots + si) * A.nref;
  }
  const bool hist = l >= A.hist_l0 && l < A.hist_l1;
  if (S->obs_w) S->obs_w += l * A.obs_step;
  if (S->obs_r) S->obs_r += l * A.obs_step;
  if (S->inj) S->inj += l * A.obs_step;
  S->hist_w = hist && S->hist_w ? S->hist_w + l * A.hist_step : nullptr;
  S->hist_r = hist && S->hist_r ? S->hist_r + l * A.hist_step : nullptr;
  S->chist_w = hist && S->chist_w ? S->chist_w + l * A.chist_step : nullptr;
  S->chist_r = hist && S->chist_r ? S->chist_r + l * A.chist_step : nullptr;
  if constexpr (M == kForward) {
    S->mask_f = phase(A, si, step, &S->src_mask);
    S->pulse.st = __dmul_rn((double)step, A.dt);
  } else if constexpr (M == kAdjoint) {
    S->mask_f = phase(A, si, step, (int*)nullptr);
    S->mask_e = phase(A, si, step - 1, (int*)nullptr);
    S->mask_c = phase(A, si, step + 1, (int*)nullptr);
  }
}

constexpr int kNeedTable = 256;

// Wait (one warp) until the items of the level before l that an item of `slab`
// depends on are complete: it reads nodes of its own slab and the two next to
// it, and overwrites values that only items there have read.  Items are
// claimed in order, so those are running or done and the wait ends whatever
// the number of resident blocks.  False on timeout or abort.
template <typename T>
__device__ __forceinline__ bool wait_level(const SweepArgs<T>& A, const int* need, int si, int slab, int l) {
  const int lane = (int)threadIdx.x & 31;
  const int dep = lane < 3 ? min(max(slab - 1 + lane, 0), A.nslab - 1) : -1;
  const unsigned* c = A.sync + 2 + (dep < 0 ? 0 : (long long)si * A.nslab + dep);
  const unsigned want = dep < 0 ? 0u : (unsigned)l * (unsigned)(dep < kNeedTable ? need[dep] : A.need[dep]);
  const long long t0 = clock64();
  for (unsigned it = 1;; ++it) {
    const bool ok = dep < 0 || load_acquire(c) >= want;
    if (__all_sync(0xffffffffu, ok)) {
      __syncwarp();
      return true;
    }
    if (A.wait < 0) return false;
    bool give_up = false;
    if ((it & 31) == 0) give_up = clock64() - t0 > A.wait || *(const volatile int*)A.err != 0;
    if (__any_sync(0xffffffffu, give_up)) return false;
  }
}

// Refined item: entries [first, end) of the slab's corner rows followed by its
// centre rows (with the transposed step's pairing of their voxels), one thread
// per row.
template <typename T, bool ADJ>
__device__ __forceinline__ void refined_item(const SweepArgs<T>& A, const Slot<T>& S, int si, int slab, int first,
                                             int end) {
  const int4 q = A.rslab[slab];
  for (int r = first + (int)threadIdx.x; r < end; r += (int)blockDim.x - kServiceThreads) {
    if (r < q.y) refined_corner<T, ADJ>(A, S, q.x + r);
    else refined_centre<T, ADJ>(A, S, q.z + (r - q.y), si);
  }
}

// Queue entry of an item for the row threads.
struct QItem {
  int si;  // -1: no more work
  int slab;
  unsigned first, end;
  int kind, zend;
};

// What bounds it and why it is built so.  FP64: the FP64 pipe (two lanes per SM
// and clock), 12.5 operations a lattice row: 131 x 118 x 143, two sources,
// 0.238 / 0.296 ms a forward / transposed level by a launch of staged tiles per
// level, 0.132 / 0.190 ms here (the pipe's floor for the forward rows: 0.093).
// Small lattices: the launches and their dependent chain, 33^3 9.0 / 16.7 us a
// level then, 6.1 / 10.7 us here.
// Two blocks of 7 row warps and a producer warp per SM leave a thread 128
// registers, which the transposed rows with their pairing need (with three
// blocks they spill: autograd's 97^3 FP64 49 us a transposed level against 44).
//
// A.nlev consecutive levels of every slot.  The blocks claim work items
// (level, slot, item) in order from one counter; an item waits until the
// previous level's items of its slab and the two next to it are complete
// (counters per slot and slab), runs, and signals its own slab.  So there is
// no launch and no device-wide barrier between levels, and blocks run into
// the next level while others finish the last.  A block's producer warp runs
// one item ahead of its row threads: it claims the item, waits for what it
// depends on, publishes it with its slot, and stages an interior item's planes.
template <typename T, StepMode M, bool TEL, bool ANI>
__global__ void __launch_bounds__(kMaxBlock + kServiceThreads, kSweepBlocksPerSm)
    sweep_kernel(const __grid_constant__ SweepArgs<T> A) {
  extern __shared__ __align__(128) unsigned char hyb_smem[];  // A.ns stages of A.nstage elements
  T* ring = reinterpret_cast<T*>(hyb_smem);
  __shared__ Slot<T> S2[2];
  __shared__ QItem Q2[2];
  __shared__ Bars B;
  __shared__ T ex[256];  // edge tiles
  __shared__ int done[2];  // row warps done with an item
  __shared__ int need[kNeedTable];  // items per slab and level
  const int t = (int)threadIdx.x, rows = (int)blockDim.x - kServiceThreads;
  for (int q = t; q < min(A.nslab, kNeedTable); q += (int)blockDim.x) need[q] = A.need[q];
  if (t == 0) {
    for (int q = 0; q < A.ns; ++q) {
      mbar_init(B.full + q, 1);
      mbar_init(B.empty + q, rows / 32);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(B.qfull + q, 2);  // the slot's copy, the item
      done[q] = 0;
      mbar_init(B.qempty + q, 1);
    }
    mbar_init_fence();
  }
  __syncthreads();
  RingPos rp = {0, 0u};
  const long long own = kOwnCycles + 64 * max(A.wait, 0LL);  // an item's waits one after the other
  if (t >= rows) {
    const int lane = t & 31;
    const unsigned per = (unsigned)A.snitems * (unsigned)A.nslots, total = per * (unsigned)A.nlev;
    auto entry = [&](unsigned it) {
      return it < total ? A.sitems[(it % per) % (unsigned)A.snitems] : make_int4(0, 0, 0, 0);
    };
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(A.sync, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    int4 q = entry(it);
    unsigned nit = 0;
    if (lane == 0) nit = atomicAdd(A.sync, 1u);
    bool ok = true;
    unsigned issued = 0;  // stages copied into
    for (int n = 0;; ++n) {
      const int b = n & 1;
      const bool more = it < total;
      const int l = (int)(it / per), si = (int)((it - (unsigned)l * per) / (unsigned)A.snitems);
      if (!mbar_wait_idle(B.qempty + b, ((n >> 1) & 1) ^ 1u, own, nullptr)) break;  // (never: items end in bounded time)
      if (!ok || !more) {
        if (lane == 0) {
          Q2[b].si = -1;
          mbar_arrive(B.qfull + b);
          mbar_arrive(B.qfull + b);
        }
        break;
      }
      if (lane == 0) {
        fence_proxy_async_shared();  // (the row threads' reads of the slot before the copy into it)
        mbar_arrive_expect_tx(B.qfull + b, (uint32_t)sizeof(Slot<T>));
        bulk_load(S2 + b, A.table + (size_t)l * A.nslots + si, (uint32_t)sizeof(Slot<T>), B.qfull + b);
      }
      nit = __shfl_sync(0xffffffffu, nit, 0);
      const int4 nq = entry(nit);  // (the next item's entry and the claim after it are on their way meanwhile)
      unsigned nnit = 0;
      if (lane == 0) nnit = atomicAdd(A.sync, 1u);
      const int kind = q.w & 255, slab = q.x;
      if (l > 0 && !wait_level(A, need, si, slab, l)) {
        if (lane == 0) atomicExch(A.err, 1);
        ok = false;
      }
      if (lane == 0) {
        Q2[b] = {si, slab, (unsigned)q.y, (unsigned)q.z, kind, q.w >> 8};
        mbar_arrive(B.qfull + b);
        if (kind == kInterior && ok) {
          fence_proxy_async_global();  // (other blocks' stores to the planes, acquired above, before the copies)
          ok = interior_produce(A, &B, ring, rp, ring_field(A, ring_slot(A, l, 0), si),
                                ring_field(A, ring_slot(A, l, 1), si), slab, q.y, A.wait, issued);
          if (!ok) atomicExch(A.err, 1);
        }
      }
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      it = nit;
      q = nq;
      nit = nnit;
    }
    // let no copy be in flight when the block exits (the row threads may have
    // given up on some): every stage issued last
    if (lane == 0) {
      for (int s = 0; s < A.ns && s < (int)min(issued, (unsigned)kMaxStages); ++s)
        mbar_wait_idle(B.full + s, s < rp.st ? rp.ph : rp.ph ^ 1u, kOwnCycles, nullptr);
    }
  } else {
    for (int n = 0;; ++n) {
      const int b = n & 1;
      if (!mbar_try(B.qfull + b, (n >> 1) & 1) && !mbar_wait_slow(B.qfull + b, (n >> 1) & 1, own, nullptr)) break;  // (never: the producer publishes in bounded time)
      const QItem q = Q2[b];
      if (q.si < 0) break;
      const Slot<T>& S = S2[b];
      if (q.kind == kInterior) {
        interior_item<T, M, TEL, ANI>(A, S, &B, ring, rp, q.si, q.slab, q.first);
      } else if (q.kind == kFace) {
        for (unsigned r = q.first + t; r < q.end; r += rows) face_entry<T, M, ANI>(A, S, q.si, q.slab, r);
      } else if (q.kind == kRefined) {
        if constexpr (!TEL && !ANI) refined_item<T, M != kForward>(A, S, q.si, q.slab, q.first, q.end);
      } else {
        const int e = (int)q.first + (t >> 7);  // one tile per 128 threads
        EdgeTile E = {-2, 0, 0, 0};
        if (e < (int)q.end) {
          const int by = (A.ny - 4 + 15) / 16, p = e - 1;
          if (q.kind == kEdgeZ) {
            const int k0 = max(1 + q.slab * A.slabz, 2), k1 = min(1 + (q.slab + 1) * A.slabz, A.nz - 2);
            E = {2, 0, k0 + 8 * e, min(k0 + 8 * e + 8, k1)};
          } else if (e == 0) {
            E = {-1, q.zend, 0, 0};
          } else if (p < by) {
            E = {1, q.zend, 2 + 16 * p, min(18 + 16 * p, A.ny - 2)};
          } else {
            E = {0, q.zend, 2 + 16 * (p - by), min(18 + 16 * (p - by), A.nx - 2)};
          }
        }
        T* sh = ex + (t & ~127);
        if constexpr (M == kAdjoint) adj_edge_tile<T, ANI>(A, S, E, t & 127, sh);
        else fwd_edge_tile<T, ANI>(A, S, E, t & 127, sh);
        if constexpr (M != kForward) {
          int i = 0, j = 0, k = 0, nf, qq[3];
          if (edge_tile_node(A, E, t & 127, i, j, k, qq, nf)) pair_if_voxel<T, ANI>(A, S, q.si, i, j, k);
        }
      }
      __syncwarp();  // the warp's stores are issued, and it is done with the slot
      // the last row warp to finish reports the item (the release takes a
      // thousand cycles and more; the others run into the next item)
      if ((t & 31) == 0) {
        __threadfence_block();
        if (atomicAdd(done + b, 1) == rows / 32 - 1) {
          __threadfence_block();
          done[b] = 0;
          mbar_arrive(B.qempty + b);
          red_release(A.sync + 2 + (long long)q.si * A.nslab + q.slab);
        }
      }
    }
  }
  // the last block leaves the counters cleared for the next launch
  __syncthreads();  // (the last item's signal is out)
  if (t == 0) {
    __threadfence();
    if (atomicAdd(A.sync + 1, 1u) == gridDim.x - 1) {
      for (int q = 0; q < 2 + A.nslots * A.nslab; ++q) A.sync[q] = 0u;
    }
  }
}

}  // namespace

template <typename T, StepMode M>
void launch_levels(const SweepArgs<T>& a, int block, int grid, int smem, cudaStream_t st) {
  if constexpr (M != kPaper) {
    if (a.ani) {
      sweep_kernel<T, M, false, true><<<grid, block + kServiceThreads, smem, st>>>(a);
      return;
    }
    if (a.sdamp) {
      sweep_kernel<T, M, true, false><<<grid, block + kServiceThreads, smem, st>>>(a);
      return;
    }
  }
  sweep_kernel<T, M, false, false><<<grid, block + kServiceThreads, smem, st>>>(a);
}

template <typename T, StepMode M>
int launch_sweep_mode(const SweepArgs<T>& a, int block, int grid, int smem, int levels, cudaStream_t st) {
  slots_kernel<T, M><<<(a.nlev * a.nslots + 127) / 128, 128, 0, st>>>(a);
  int n = 1;
  const int parts = a.nlev / levels > 1 ? a.nlev / levels : 1;  // (even ones: short launches cost most)
  levels = (a.nlev + parts - 1) / parts;
  SweepArgs<T> b = a;
  for (int l = 0; l < a.nlev; l += b.nlev, ++n) {
    b.table = a.table + (size_t)l * a.nslots;
    b.ring0 = (a.ring0 + a.dir * (l % 3) + 3) % 3;
    b.nlev = a.nlev - l < levels ? a.nlev - l : levels;
    launch_levels<T, M>(b, block, grid, smem, st);
  }
  return n;
}

int launch_sweep(const SweepArgs<double>& a, StepMode mode, int block, int grid, int smem, int levels,
                 cudaStream_t st) {
  if (mode == kForward) return launch_sweep_mode<double, kForward>(a, block, grid, smem, levels, st);
  if (mode == kAdjoint) return launch_sweep_mode<double, kAdjoint>(a, block, grid, smem, levels, st);
  return launch_sweep_mode<double, kPaper>(a, block, grid, smem, levels, st);
}

template <typename T, StepMode M, bool TEL, bool ANI>
int variant_occupancy(int block, int smem) {
  int n = 0;
  if (cudaFuncSetAttribute(sweep_kernel<T, M, TEL, ANI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxRing) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sweep_kernel<T, M, TEL, ANI>, block + kServiceThreads, smem) !=
          cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return n;
}

int sweep_blocks_per_sm(int block, int smem) {
  int n = variant_occupancy<double, kForward, false, false>(block, smem);
  auto least = [&n](int q) { n = q < n ? q : n; };
  least(variant_occupancy<double, kAdjoint, false, false>(block, smem));
  least(variant_occupancy<double, kPaper, false, false>(block, smem));
  least(variant_occupancy<double, kForward, true, false>(block, smem));
  least(variant_occupancy<double, kAdjoint, true, false>(block, smem));
  least(variant_occupancy<double, kForward, false, true>(block, smem));
  least(variant_occupancy<double, kAdjoint, false, true>(block, smem));
  return n > 0 ? n : 1;
}

}  // namespace hyb
