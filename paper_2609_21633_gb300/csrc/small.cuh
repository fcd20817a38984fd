// A apply on the coarse multigrid levels (N <= 16), element-parallel (included by kernels.cu inside its
// namespace, after the element ops, the epilogue and project_vec).
//
// A streaming tile kernel gives such a level 10 tile columns, each a serial radial sweep: on level 4 / 17
// layers the FP64 apply ran 20 CTAs on 152 SMs (229 us; 25 us per layer of one SM's FP64 pipe).  Here every
// cell has a thread (every wedge three, FP64), is computed once and leaves its contributions in a scratch array (in
// L2); a second kernel gathers every copy of a node from the elements of its diamond, sums the copies by shuffles
// -- no interface pass -- and runs the fused vector update at every copy.
// The same two device functions carry the coarsest-level conjugate gradients (k_cg_cluster below).
// Bound by latency (two dependent launches of a few microseconds), in FP64 by the FP64 pipes (64 cycles
// per instruction of a warp on an SM partition).  V-cycles went from (streaming tiles filling the SMs) 1017
// to 334 us (FP32, level 4 / 17 layers), 1404 to 594 us (FP32, two radial points, 5 / 33) and 3999 to 1521 us (FP64,
// 5 / 33); a thread per group that walks its copies, instead of one per copy, left them at 703, 1072 and 2816 us.
// Sums run in a fixed order (copies in ascending layout order; the six triangles; bottom then top
// contributions), so results do not depend on scheduling.

struct SmallDims {
  int N, n_r, P, ls, ds, nll;  // ls / ds: layer / diamond stride of the node layout, nll: lateral layout size
  int ncell, npad, n_groups;   // cells, lateral points (every copy) rounded up to whole warps, interface groups
  int div_term;
  double hgc;  // kappa (3 + c) / 18 of the hourglass control
  Points pts;
  template <typename T>
  __device__ __forceinline__ T hgk() const { return (T)hgc; }
};
inline SmallDims small_dims(const Level& L, int div_term, double hgc) {
  SmallDims s;
  s.N = L.N, s.n_r = L.n_r, s.P = L.P, s.ls = (int)L.layer_stride, s.ds = (int)L.diamond_stride;
  s.nll = (int)L.n_lat_layout;
  s.ncell = 10 * L.N * L.N * (L.n_r - 1);
  s.pts = points_of(L);
  s.npad = (s.pts.n + 31) / 32 * 32, s.n_groups = L.n_groups, s.div_term = div_term, s.hgc = hgc;
  return s;
}

template <typename T>
struct SmallTab {  // tables of the level in its precision
  const T *geo, *lay, *svec, *gs;
  EtaView<T> eta;
  int bc_in, bc_out;
};
template <typename T>
inline SmallTab<T> small_tab(const Level& L, BC bc) {
  return SmallTab<T>{Tab<T>::geo(L), Tab<T>::lay(L), Tab<T>::s(L), Tab<T>::gs(L), etav<T>(L), bc.in, bc.out};
}

// How a level's elements are spread: three threads per wedge in FP64, where a cell's chain of instructions bounds the
// small levels (level 3 / 9 layers: 8.5 against 13 us, FP64 V-cycle level 5 / 33 1521 against 1756 us), one thread per
// cell in FP32, where the extra contributions cost more than the shorter chain saves (V-cycle level 4 / 17 layers
// 381 to 388 against 366 us).
template <typename T>
constexpr bool kSmallWedges = sizeof(T) == 8;
static_assert(small_values<double>() == (kSmallWedges<double> ? 36 : 24), "scratch of a cell");
static_assert(small_values<float>() == (kSmallWedges<float> ? 36 : 24), "scratch of a cell");

// FP64: contributions of the wedges to their six nodes, thread per wedge and component: three neighbouring lanes share a
// wedge, ten wedges a warp (two lanes idle).  A lane forms its component's row of the strain, exchanges the transposed
// entries and the trace by shuffles and contracts its row of the stress: about 45 dependent FP64 instructions
// instead of the 265 of a thread per cell (13 us of latency on every small level).  The rows of M^-1 and of the strain
// are held in the order c, c + 1, c + 2 (mod 3) of the lane's component c, so no register is indexed by c.
// HG: hourglass control, Q2: the second radial point (see OpA, OpA2).  Wedge v of wb .. wb + 9 (wedge layout); its
// local node a, component c gets sc[(3 a + c) nw + v] at the bottom and sc[(9 + 3 a + c) nw + v] at the top.  CG: loads
// bypass L1 (the input was written by other SMs within the same kernel).  All lanes of the warp call it.
template <typename T, bool HG, bool Q2, bool CG>
__device__ __forceinline__ void small_wedges(const SmallDims& S, const SmallTab<T>& B, const T* const (&in)[3], int wb,
                                             T* __restrict__ sc) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = (int)threadIdx.x & 31, g = lane / 3, c = lane - 3 * g, base = 3 * g, nw = 2 * S.ncell;
  const int v = min(wb + min(g, 9), nw - 1);  // idle lanes repeat the last wedge
  const bool live = g < 10 && wb + g < nw;
  const int N = S.N, nc = S.n_r - 1;
  const int w = v & 1, cell = v >> 1, j = cell % N, r0 = cell / N, i = r0 % N, r1 = r0 / N, k = r1 % nc, d = r1 / nc;
  const int t = ((d * N + i) * N + j) * 2 + w, nt = 20 * N * N;
  const int lat = d * S.ls + i * S.P + j, o = lat + d * (S.ds - S.ls) + k * S.ls;
  // local nodes 0, 1, 2: W0 (i, j), (i + 1, j), (i, j + 1); W1 (i + 1, j + 1), (i, j + 1), (i + 1, j)
  const int del[3] = {w ? S.P + 1 : 0, w ? 1 : S.P, w ? S.P : 1};
  const T* const u = c == 0 ? in[0] : (c == 1 ? in[1] : in[2]);
  T b[3], tp[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    b[a] = CG ? __ldcg(u + o + del[a]) : u[o + del[a]];
    tp[a] = CG ? __ldcg(u + o + S.ls + del[a]) : u[o + S.ls + del[a]];
  }
  const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
  T M[3][3];  // M[m][r] = M^-1[m, c + r]
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    M[m][0] = B.geo[(3 * m + c) * nt + t], M[m][1] = B.geo[(3 * m + c1) * nt + t], M[m][2] = B.geo[(3 * m + c2) * nt + t];
  }
  const T dM = B.geo[9 * nt + t], e = eta_at(B.eta, (int64_t)v, (int64_t)t);
  const T* const lc = B.lay + kLayerStride * k;
  const T r = lc[4], ve = lc[5] * dM * e;
  // boundary projection: v_c -= (v . s) s_c, the dot product over the three lanes
  auto project = [&](T (&x)[3], bool here, int bc) {
    if (!__any_sync(kAll, here)) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const T s = B.svec[c * S.nll + lat + del[a]], q = x[a] * s;
      const T dot = (__shfl_sync(kAll, q, base) + __shfl_sync(kAll, q, base + 1)) + __shfl_sync(kAll, q, base + 2);
      if (here) x[a] = bc == TN_BC_NOSLIP ? (T)0 : x[a] - dot * s;
    }
  };
  project(b, k == 0, B.bc_in);
  project(tp, k == nc - 1, B.bc_out);
  const T d0 = tp[0] - b[0], d1 = tp[1] - b[1], d2 = tp[2] - b[2];
  const T ax = (tp[1] + b[1]) - (tp[0] + b[0]), ay = (tp[2] + b[2]) - (tp[0] + b[0]), az = (d0 + d1) + d2;
  // stress row of a strain row G: f (G + G^T) - 2/3 f tr G on the diagonal
  auto stress = [&](const T (&G)[3], T f, T (&R)[3]) {
    const T g1 = __shfl_sync(kAll, G[2], base + c1), g2 = __shfl_sync(kAll, G[1], base + c2);  // G^T entries
    R[0] = (f + f) * G[0];
    if (S.div_term) {
      const T tr = (__shfl_sync(kAll, G[0], base) + __shfl_sync(kAll, G[0], base + 1)) + __shfl_sync(kAll, G[0], base + 2);
      R[0] += (f * (T)(-2.0 / 3.0)) * tr;
    }
    R[1] = f * (G[1] + g1), R[2] = f * (G[2] + g2);
  };
  auto dot = [&](const T (&R)[3], int m) { return R[0] * M[m][0] + R[1] * M[m][1] + R[2] * M[m][2]; };
  T G[3], R[3];
  const T azr = az * r;
#pragma unroll
  for (int x = 0; x < 3; ++x) G[x] = ax * M[0][x] + ay * M[1][x] + azr * M[2][x];
  stress(G, ve, R);
  T h0 = dot(R, 0), h1 = dot(R, 1);
  const T h2 = r * dot(R, 2);
  T y0 = h2, y1 = h2, y2 = h2;
  if constexpr (HG) {
    T l = 0, q = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const T s01 = M[0][x] + M[1][x];
      l += s01 * s01 + M[0][x] * M[0][x] + M[1][x] * M[1][x];
      q += M[2][x] * M[2][x];
    }
    const T k9 = lc[8], a3 = az * (T)(1.0 / 3.0);
    const T al1 = (d1 - a3) - k9 * (ax + ax - ay), al2 = (d2 - a3) - k9 * (ay + ay - ax);
    const T eps = (S.template hgk<T>() * e) * (lc[5] * ((T)2 * dM * l) + lc[9] * ((T)6 * dM * q));
    const T ek = eps * k9, e3 = eps * (T)(1.0 / 3.0);
    const T b1 = (al1 + al1) - al2, b2 = (al2 + al2) - al1;
    h0 -= ek * b1, h1 -= ek * b2;
    const T v1 = e3 * b1, v2 = e3 * b2;
    y0 -= v1 + v2, y1 += v1, y2 += v2;
  }
  if constexpr (Q2) {
    const T bx = d1 - d0, by = d2 - d0, a3 = az * (T)(1.0 / 3.0);
    T G1[3], R1[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) G1[x] = bx * M[0][x] + by * M[1][x] + a3 * M[2][x];
    stress(G1, ve * (T)(1.0 / 3.0), R1);
    const T k0 = dot(R1, 0), k1 = dot(R1, 1), k2 = dot(R1, 2) * (T)(1.0 / 3.0);
    y0 += k2 - (k0 + k1), y1 += k2 + k0, y2 += k2 + k1;
  }
  if (!live) return;
  const T x0 = -(h0 + h1);
  T* const q = sc + v;
  q[c * nw] = x0 - y0, q[(3 + c) * nw] = h0 - y1, q[(6 + c) * nw] = h1 - y2;
  q[(9 + c) * nw] = x0 + y0, q[(12 + c) * nw] = h0 + y1, q[(15 + c) * nw] = h1 + y2;
}

// Partial sum of the wedges of diamond d around node (i, j, k).
template <typename T>
__device__ __forceinline__ void small_gather(const SmallDims& S, const T* __restrict__ sc, int d, int i, int j, int k,
                                             T (&v)[3]) {
  const int N = S.N, nc = S.n_r - 1, nw = 2 * S.ncell;
  // cell offset, wedge and local node of the six triangles around a node
  constexpr int tri[6][4] = {{0, 0, 0, 0}, {-1, 0, 0, 1}, {-1, 0, 1, 2}, {0, -1, 0, 2}, {0, -1, 1, 1}, {-1, -1, 1, 0}};
  T a[12][3];  // all loads issued before the sums; absent wedges count 0
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int ci = i + tri[q][0], cj = j + tri[q][1];
    const bool ok = ci >= 0 && cj >= 0 && ci < N && cj < N;
    const int vb = (((d * nc + k) * N + ci) * N + cj) * 2 + tri[q][2], vt = vb - 2 * N * N;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      a[q][x] = ok && k < nc ? __ldcg(sc + (3 * tri[q][3] + x) * nw + vb) : (T)0;
      a[6 + q][x] = ok && k > 0 ? __ldcg(sc + (9 + 3 * tri[q][3] + x) * nw + vt) : (T)0;
    }
  }
#pragma unroll
  for (int x = 0; x < 3; ++x)
    v[x] += (((a[0][x] + a[1][x]) + (a[2][x] + a[3][x])) + (a[4][x] + a[5][x])) +
            (((a[6][x] + a[7][x]) + (a[8][x] + a[9][x])) + (a[10][x] + a[11][x]));
}

// FP32, thread per cell: contributions of cell c = ((d (n_r - 1) + k) N + i) N + j to its eight nodes: bottom corner q, component x
// at sc[(3 q + x) ncell + c], top at sc[(12 + 3 q + x) ncell + c].  CG loads bypass L1 when the input was
// written by other SMs within the same kernel.
template <typename T, typename Op, bool CG>
__device__ __forceinline__ void small_cell(const SmallDims& S, const SmallTab<T>& B, const Op& op, const T* const (&in)[3],
                                           int c, T* __restrict__ sc) {
  const int N = S.N, nc = S.n_r - 1;
  const int j = c % N, r0 = c / N, i = r0 % N, r1 = r0 / N, k = r1 % nc, d = r1 / nc;
  const int t0 = ((d * N + i) * N + j) * 2, nt = 20 * N * N;
  const int o = d * S.ds + k * S.ls + i * S.P + j, lat = d * S.ls + i * S.P + j;
  const int del[4] = {0, S.P, 1, S.P + 1};
  T s[4][3], dd[4][3];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    T b[3], t[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      b[x] = CG ? __ldcg(in[x] + o + del[q]) : in[x][o + del[q]];
      t[x] = CG ? __ldcg(in[x] + o + S.ls + del[q]) : in[x][o + S.ls + del[q]];
    }
    if (k == 0) project_vec(b, B.svec, (int64_t)lat + del[q], (int64_t)S.nll, B.bc_in);
    if (k == nc - 1) project_vec(t, B.svec, (int64_t)lat + del[q], (int64_t)S.nll, B.bc_out);
#pragma unroll
    for (int x = 0; x < 3; ++x) s[q][x] = b[x] + t[x], dd[q][x] = t[x] - b[x];
  }
  T Mi[2][9], dM[2], e[2];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
#pragma unroll
    for (int q = 0; q < 9; ++q) Mi[w][q] = B.geo[q * nt + t0 + w];
    dM[w] = B.geo[9 * nt + t0 + w];
    e[w] = eta_at(B.eta, (int64_t)2 * c + w, (int64_t)t0 + w);
  }
  const typename Op::Col col = op.column(Mi, dM, t0);
  T ab[4][3], at[4][3];
  op.cell(s, dd, Mi, dM, B.lay + kLayerStride * k, e, ab, at, col);
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      sc[(3 * q + x) * S.ncell + c] = ab[q][x];
      sc[(12 + 3 * q + x) * S.ncell + c] = at[q][x];
    }
}

// Partial sum of the cells of diamond d around node (i, j, k).
template <typename T>
__device__ __forceinline__ void small_gather_cells(const SmallDims& S, const T* __restrict__ sc, int d, int i, int j, int k,
                                             T (&v)[3]) {
  const int N = S.N, nc = S.n_r - 1;
  const int di[4] = {0, 1, 0, 1}, dj[4] = {0, 0, 1, 1};
  T a[8][3];  // all loads issued before the sums; absent cells count 0
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ci = i - di[q], cj = j - dj[q];
    const bool ok = ci >= 0 && cj >= 0 && ci < N && cj < N;
    const int cb = ((d * nc + k) * N + ci) * N + cj, ct = cb - N * N;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      a[q][x] = ok && k < nc ? __ldcg(sc + (3 * q + x) * S.ncell + cb) : (T)0;
      a[4 + q][x] = ok && k > 0 ? __ldcg(sc + (12 + 3 * q + x) * S.ncell + ct) : (T)0;
    }
  }
#pragma unroll
  for (int x = 0; x < 3; ++x)
    v[x] += ((a[0][x] + a[1][x]) + (a[2][x] + a[3][x])) + ((a[4][x] + a[5][x]) + (a[6][x] + a[7][x]));
}

// y = (P A P + I - P) in at node layer k of point p from the cells' contributions, the same at every copy; o: the
// copy's layout offset, u: its warp's first point.  All lanes of the warp call it.
template <typename T, bool CG>
__device__ __forceinline__ void small_node(const SmallDims& S, const SmallTab<T>& B, const T* const (&in)[3],
                                           const T* __restrict__ sc, const Point& p, int u, int k, int o, T (&v)[3]) {
  v[0] = v[1] = v[2] = (T)0;
  T w[3] = {0, 0, 0};
  const bool surface = k == 0 || k == S.n_r - 1;
  if (p.cnt) {
    if (surface)
#pragma unroll
      for (int x = 0; x < 3; ++x) w[x] = CG ? __ldcg(in[x] + o) : in[x][o];
    if constexpr (kSmallWedges<T>) small_gather(S, sc, p.d, p.i, p.j, k, v);
    else small_gather_cells(S, sc, p.d, p.i, p.j, k, v);
  }
  copies_sum<T, 3>(p, u, v);
  if (surface && p.cnt) {
    if ((k == 0 ? B.bc_in : B.bc_out) == TN_BC_NOSLIP) {
#pragma unroll
      for (int x = 0; x < 3; ++x) v[x] = w[x];
    } else {
      T s[3];
      point_dir(p, B.gs, S.n_groups, B.svec, S.ls, S.P, S.nll, s);
      const T dv = (w[0] - v[0]) * s[0] + (w[1] - v[1]) * s[1] + (w[2] - v[2]) * s[2];
#pragma unroll
      for (int x = 0; x < 3; ++x) v[x] += dv * s[x];
    }
  }
}

constexpr int kSmallBlock = 64;  // 20 wedges or 64 cells: short CTAs spread a level evenly over the SMs

template <typename T, bool HG, bool Q2>
__global__ void __launch_bounds__(kSmallBlock) k_small_wedge(SmallDims S, SmallTab<T> B, const T* __restrict__ in0,
                                                             const T* __restrict__ in1, const T* __restrict__ in2,
                                                             T* __restrict__ sc) {
  const int wb = ((int)(blockIdx.x * kSmallBlock + threadIdx.x) >> 5) * 10;
  if (wb >= 2 * S.ncell) return;
  const T* const in[3] = {in0, in1, in2};
  small_wedges<T, HG, Q2, false>(S, B, in, wb, sc);
}

template <typename T, typename Op>
__global__ void __launch_bounds__(kSmallBlock) k_small_cell(SmallDims S, SmallTab<T> B, Op op, const T* __restrict__ in0,
                                                            const T* __restrict__ in1, const T* __restrict__ in2,
                                                            T* __restrict__ sc) {
  const int c = blockIdx.x * kSmallBlock + threadIdx.x;
  if (c >= S.ncell) return;
  const T* const in[3] = {in0, in1, in2};
  small_cell<T, Op, false>(S, B, op, in, c, sc);
}

// The element op of a level's variant (FP32).
template <typename T, bool HG, bool Q2>
struct SmallOp {
  static __host__ __device__ __forceinline__ OpA<T, HG> make(const SmallDims& S) { return OpA<T, HG>{S.div_term, (T)S.hgc}; }
};
template <typename T, bool HG>
struct SmallOp<T, HG, true> {
  static __host__ __device__ __forceinline__ OpA2<T> make(const SmallDims& S) { return OpA2<T>{S.div_term}; }
};

template <typename T, int EPI>
__global__ void __launch_bounds__(128) k_small_node(SmallDims S, SmallTab<T> B, const T* __restrict__ in0,
                                                    const T* __restrict__ in1, const T* __restrict__ in2,
                                                    const T* __restrict__ sc, T* __restrict__ out0, T* __restrict__ out1,
                                                    T* __restrict__ out2, EpiArgs<T> E) {
  const int u = blockIdx.x * 128 + threadIdx.x, k = blockIdx.y;  // grid: points x layers
  const Point p = point_at(S.pts, u);
  const T* const in[3] = {in0, in1, in2};
  const int o = p.d * S.ds + k * S.ls + p.i * S.P + p.j;
  EpiOps<T, EPI> ops;
  if (p.cnt) ops.load(E, in0, in1, in2, o);
  T v[3];
  small_node<T, false>(S, B, in, sc, p, u & ~31, k, o, v);
  if (!p.cnt) return;
  if (EPI != EPI_NONE) {
    ops.apply(E, o, v);
  } else {
    out0[o] = v[0], out1[o] = v[1], out2[o] = v[2];
  }
}

// ---------------------------------------------------------------- coarsest-level conjugate gradients
// The whole block-Jacobi-preconditioned CG of the coarsest level (Sec. 7) in one launch of one cluster of
// eight CTAs: the kernel-per-step form took three launches per step, about 150 in a captured V-cycle, each
// of them a few microseconds of latency for a level of some hundred nodes.  Every copy of a node has its thread,
// which keeps the copy's r, z, x, p (the copies of a node compute the same bits; the first one counts in the inner
// products): in registers when the level has at most one node per thread, else in memory.  Cells and nodes go
// round the CTAs warp by warp; data of other SMs (p, the cells' contributions) is read past L1 after a cluster
// barrier (release / acquire).  Sums: a thread's products in FP64, then warps, CTA and the eight CTAs in a
// fixed order, every thread the same result, so the stopping test is uniform.
constexpr int kCgCtas = 8, kCgThreads = 256;

template <typename T>
struct CgArgs {
  const T *b0, *b1, *b2;  // right-hand side (layout)
  T *x[3], *r[3], *z[3], *p[3];
  const T* binv[6];
  const T* rad;  // node radii (rotation projection)
  T* sc;
  double ginv[9];  // inverse rotation Gram matrix
  double tol2;
  int maxit, project;
};

template <typename T, bool HG, bool Q2, bool ONE>
__global__ void __launch_bounds__(kCgThreads) k_cg_cluster(SmallDims S, SmallTab<T> B, CgArgs<T> A) {
  namespace cgr = cooperative_groups;
  cgr::cluster_group cl = cgr::this_cluster();
  __shared__ double wsum[kCgThreads / 32][3], csum[2][kCgCtas][3];
  const int rank = (int)cl.block_rank();
  const int gt = (((int)threadIdx.x >> 5) * kCgCtas + rank) * 32 + ((int)threadIdx.x & 31);
  constexpr int GT = kCgCtas * kCgThreads;
  const int nn = S.npad * S.n_r;  // a multiple of 32: warps enter the loops over nodes whole
  int par = 0;
  // sum of up to three values over the cluster; ends with a cluster barrier, which also publishes global writes
  auto total = [&](double (&a)[3], int n) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int c = 0; c < n; ++c) {
      double s = a[c];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) wsum[wid][c] = s;
    }
    __syncthreads();
    if (threadIdx.x < kCgCtas) {
      double* dst = cl.map_shared_rank(&csum[par][0][0], (unsigned)threadIdx.x) + 3 * rank;
      for (int c = 0; c < n; ++c) {
        double s = 0.0;
        for (int w = 0; w < kCgThreads / 32; ++w) s += wsum[w][c];
        dst[c] = s;
      }
    }
    cl.sync();
    for (int c = 0; c < n; ++c) {
      double s = 0.0;
      for (int q = 0; q < kCgCtas; ++q) s += csum[par][q][c];
      a[c] = s;
    }
    par ^= 1;  // the next sum's remote writes go to the other buffer: it is read two barriers later
  };
  // a thread's node: copy, layer, offsets, and its vectors (registers when ONE)
  struct Node {
    Point p;
    int u, k, o;
    T x[3], r[3], z[3], q[3], b[6], d[3];  // q: search direction; b: D^-1; d: unit direction times the radius
  };
  Node one;
  auto locate = [&](int t, Node& n) {
    n.k = t / S.npad, n.u = t - n.k * S.npad;
    n.p = point_at(S.pts, n.u);
    n.o = n.p.d * S.ds + n.k * S.ls + n.p.i * S.P + n.p.j;
    if (!n.p.cnt) return;
#pragma unroll
    for (int q = 0; q < 6; ++q) n.b[q] = A.binv[q][n.o];
    if (A.project) {
      T s[3];
      point_dir(n.p, B.gs, S.n_groups, B.svec, S.ls, S.P, S.nll, s);
#pragma unroll
      for (int c = 0; c < 3; ++c) n.d[c] = s[c];
    }
  };
  auto load = [&](T* const (&a)[3], const Node& n, T (&v)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = a[c][n.o];
  };
  auto store = [&](T* const (&a)[3], const Node& n, const T (&v)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c][n.o] = v[c];
  };
  // f over this thread's nodes (whole warps, unused lanes with cnt = 0)
  auto each = [&](auto&& f) {
    if constexpr (ONE) {
      if (gt < nn) f(one);
    } else {
      for (int t = gt; t < nn; t += GT) {
        Node n;
        locate(t, n);
        f(n);
      }
    }
  };
  auto counts = [&](const Node& n) { return n.p.cnt > 0 && n.p.lane == 0; };
  auto bmul3 = [&](const Node& n, const T (&r)[3], T (&z)[3]) {
    z[0] = n.b[0] * r[0] + n.b[3] * r[1] + n.b[4] * r[2];
    z[1] = n.b[3] * r[0] + n.b[1] * r[1] + n.b[5] * r[2];
    z[2] = n.b[4] * r[0] + n.b[5] * r[1] + n.b[2] * r[2];
  };
  // rotation component w = Ginv (sum over nodes of x cross v), removed as v - w cross x
  auto spin = [&](const Node& n, const T (&v)[3], double (&a)[3]) {
    const double r = A.rad[n.k], x[3] = {r * n.d[0], r * n.d[1], r * n.d[2]}, y[3] = {v[0], v[1], v[2]};
    a[0] += x[1] * y[2] - x[2] * y[1];
    a[1] += x[2] * y[0] - x[0] * y[2];
    a[2] += x[0] * y[1] - x[1] * y[0];
  };
  auto omega = [&](double (&a)[3], double (&w)[3]) {
    total(a, 3);
    for (int c = 0; c < 3; ++c) w[c] = A.ginv[3 * c] * a[0] + A.ginv[3 * c + 1] * a[1] + A.ginv[3 * c + 2] * a[2];
  };
  auto despin = [&](const Node& n, const double (&w)[3], T (&v)[3]) {
    const double r = A.rad[n.k], x[3] = {r * n.d[0], r * n.d[1], r * n.d[2]};
    v[0] -= (T)(w[1] * x[2] - w[2] * x[1]);
    v[1] -= (T)(w[2] * x[0] - w[0] * x[2]);
    v[2] -= (T)(w[0] * x[1] - w[1] * x[0]);
  };

  if constexpr (ONE)
    if (gt < nn) locate(gt, one);
  // A CTA's shared memory may be written by the others only once it runs: total() stores to all eight before its own
  // barrier, so the cluster meets here first (one barrier per launch, behind the loads above).
  cl.sync();
  double w[3] = {0, 0, 0}, acc[3] = {0, 0, 0};
  if (A.project) {
    each([&](Node& n) {
      if (!counts(n)) return;
      const T b[3] = {A.b0[n.o], A.b1[n.o], A.b2[n.o]};
      spin(n, b, acc);
    });
    omega(acc, w);
  }
  // r = b (rotations removed), z = D^-1 r, p = z, x = 0
  acc[0] = 0.0;
  each([&](Node& n) {
    if (!n.p.cnt) return;
    n.r[0] = A.b0[n.o], n.r[1] = A.b1[n.o], n.r[2] = A.b2[n.o];
    if (A.project) despin(n, w, n.r);
    bmul3(n, n.r, n.z);
    T d = (T)0;
#pragma unroll
    for (int c = 0; c < 3; ++c) n.x[c] = (T)0, n.q[c] = n.z[c], d += n.r[c] * n.z[c];
    if (counts(n)) acc[0] += (double)d;
    store(A.p, n, n.q);
    if (!ONE) store(A.r, n, n.r), store(A.x, n, n.x);
  });
  total(acc, 1);
  const double rz0 = acc[0];
  double rz = rz0;
  const T* const pp[3] = {A.p[0], A.p[1], A.p[2]};
  if (rz0 > 0.0) {
    for (int it = 0; it < A.maxit; ++it) {
      if constexpr (kSmallWedges<T>) {
        for (int wb = (gt >> 5) * 10; wb < 2 * S.ncell; wb += (GT / 32) * 10) small_wedges<T, HG, Q2, true>(S, B, pp, wb, A.sc);
      } else {
        const auto op = SmallOp<T, HG, Q2>::make(S);
        for (int c = gt; c < S.ncell; c += GT) small_cell<T, decltype(op), true>(S, B, op, pp, c, A.sc);
      }
      cl.sync();
      acc[0] = 0.0;
      each([&](Node& n) {  // z holds q = K p until the update
        small_node<T, true>(S, B, pp, A.sc, n.p, n.u & ~31, n.k, n.o, n.z);
        if (!n.p.cnt) return;
        if (!ONE) load(A.p, n, n.q), store(A.z, n, n.z);
        T d = (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) d += n.q[c] * n.z[c];
        if (counts(n)) acc[0] += (double)d;
      });
      total(acc, 1);
      const T al = (T)(rz / acc[0]);
      acc[0] = 0.0;
      each([&](Node& n) {
        if (!n.p.cnt) return;
        if (!ONE) load(A.x, n, n.x), load(A.r, n, n.r), load(A.p, n, n.q), load(A.z, n, n.z);
#pragma unroll
        for (int c = 0; c < 3; ++c) n.x[c] += al * n.q[c], n.r[c] -= al * n.z[c];
        bmul3(n, n.r, n.z);
        T d = (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) d += n.r[c] * n.z[c];
        if (counts(n)) acc[0] += (double)d;
        if (!ONE) store(A.x, n, n.x), store(A.r, n, n.r), store(A.z, n, n.z);
      });
      total(acc, 1);
      const double rzn = acc[0];
      if (!(rzn > A.tol2 * rz0) || it == A.maxit - 1) break;
      const T be = (T)(rzn / rz);
      rz = rzn;
      each([&](Node& n) {
        if (!n.p.cnt) return;
        if (!ONE) load(A.p, n, n.q), load(A.z, n, n.z);
#pragma unroll
        for (int c = 0; c < 3; ++c) n.q[c] = n.z[c] + be * n.q[c];
        store(A.p, n, n.q);
      });
      cl.sync();
    }
  }
  // x (rotations removed)
  acc[0] = acc[1] = acc[2] = 0.0;
  if (A.project) {
    each([&](Node& n) {
      if (!counts(n)) return;
      if (!ONE) load(A.x, n, n.x);
      spin(n, n.x, acc);
    });
    omega(acc, w);
  }
  each([&](Node& n) {
    if (!n.p.cnt) return;
    if (!ONE) load(A.x, n, n.x);
    if (A.project) despin(n, w, n.x);
    store(A.x, n, n.x);
  });
  cl.sync();  // no CTA leaves while another may still write its shared memory
}
