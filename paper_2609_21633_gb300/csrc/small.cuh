// A apply on the coarse multigrid levels (N <= 16), cell-parallel (included by kernels.cu inside its
// namespace, after the element ops, the epilogue and project_vec).
//
// A streaming tile kernel gives such a level 10 tile columns, each a serial radial sweep: on level 4 / 17
// layers the FP64 apply ran 20 CTAs on 152 SMs (229 us; 25 us per layer of one SM's FP64 pipe).  Here every
// cell is its own thread, computed once, and leaves its 24 corner contributions in a scratch array (about
// 200 bytes per cell, in L2); a second kernel gathers every copy of a node from the cells of its diamond, sums the
// copies by shuffles -- no interface pass -- and runs the fused vector update at every copy.
// The same two device functions carry the coarsest-level conjugate gradients (k_cg_cluster below).
// Bound by latency (two dependent launches of a few microseconds), in FP64 by the FP64 pipes (a cell's chain of
// about 265 instructions at 64 cycles each on an SM partition).  V-cycles went from (streaming tiles filling the SMs) 1017
// to 366 us (FP32, level 4 / 17 layers), 1404 to 647 us (FP32, two radial points, 5 / 33) and 3999 to 1756 us (FP64,
// 5 / 33); a thread per group that walks its copies, instead of one per copy, left them at 703, 1072 and 2816 us.
// Sums run in a fixed order (copies in ascending layout order; corners 00, 10, 01, 11; bottom then top
// contributions), so results do not depend on scheduling.

struct SmallDims {
  int N, n_r, P, ls, ds, nll;  // ls / ds: layer / diamond stride of the node layout, nll: lateral layout size
  int ncell, npad, n_groups;   // cells, lateral points (every copy) rounded up to whole warps, interface groups
  Points pts;
};
inline SmallDims small_dims(const Level& L) {
  SmallDims s;
  s.N = L.N, s.n_r = L.n_r, s.P = L.P, s.ls = (int)L.layer_stride, s.ds = (int)L.diamond_stride;
  s.nll = (int)L.n_lat_layout;
  s.ncell = 10 * L.N * L.N * (L.n_r - 1);
  s.pts = points_of(L);
  s.npad = (s.pts.n + 31) / 32 * 32, s.n_groups = L.n_groups;
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

// Contributions of cell c = ((d (n_r - 1) + k) N + i) N + j to its eight nodes: bottom corner q, component x
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
__device__ __forceinline__ void small_gather(const SmallDims& S, const T* __restrict__ sc, int d, int i, int j, int k,
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
    small_gather(S, sc, p.d, p.i, p.j, k, v);
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

constexpr int kSmallBlock = 64;  // threads per CTA: 32 FP64 lanes of a warp take 16 cycles per instruction on an
                                 // SM's FP64 pipe, so short CTAs spread a level's cells evenly over the SMs

template <typename T, typename Op>
__global__ void __launch_bounds__(kSmallBlock) k_small_cell(SmallDims S, SmallTab<T> B, Op op, const T* __restrict__ in0,
                                                            const T* __restrict__ in1, const T* __restrict__ in2,
                                                            T* __restrict__ sc) {
  const int c = blockIdx.x * kSmallBlock + threadIdx.x;
  if (c >= S.ncell) return;
  const T* const in[3] = {in0, in1, in2};
  small_cell<T, Op, false>(S, B, op, in, c, sc);
}

template <typename T, int EPI>
__global__ void __launch_bounds__(128) k_small_node(SmallDims S, SmallTab<T> B, const T* __restrict__ in0,
                                                    const T* __restrict__ in1, const T* __restrict__ in2,
                                                    const T* __restrict__ sc, T* __restrict__ out0, T* __restrict__ out1,
                                                    T* __restrict__ out2, EpiArgs<T> E) {
  const int u = blockIdx.x * 128 + threadIdx.x, k = blockIdx.y;  // grid: points x layers
  const Point p = point_at(S.pts, u);
  const T* const in[3] = {in0, in1, in2};
  const int o = p.d * S.ds + k * S.ls + p.i * S.P + p.j;
  if (p.cnt) epi_prefetch<T, EPI>(E, o);
  T v[3];
  small_node<T, false>(S, B, in, sc, p, u & ~31, k, o, v);
  if (!p.cnt) return;
  if (EPI != EPI_NONE) {
    epilogue<T, EPI>(E, in0, in1, in2, o, v);
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

template <typename T, typename Op, bool ONE>
__global__ void __launch_bounds__(kCgThreads) k_cg_cluster(SmallDims S, SmallTab<T> B, Op op, CgArgs<T> A) {
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
      for (int c = gt; c < S.ncell; c += GT) small_cell<T, Op, true>(S, B, op, pp, c, A.sc);
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
