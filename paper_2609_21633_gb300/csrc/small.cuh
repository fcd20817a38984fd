// A apply on the coarse multigrid levels (N <= 16), cell-parallel (included by kernels.cu inside its
// namespace, after the element ops, the epilogue and project_vec).
//
// A streaming tile kernel gives such a level 10 tile columns, each a serial radial sweep: on level 4 / 17
// layers the FP64 apply ran 20 CTAs on 152 SMs (229 us; 25 us per layer of one SM's FP64 pipe).  Here every
// cell is its own thread, computed once, and leaves its 24 corner contributions in a scratch array (about
// 200 bytes per cell, in L2); a second kernel gathers every unique node from the cells around it -- over all
// diamonds that share it, so there is no interface pass -- and runs the fused vector update at every copy.
// The same two device functions carry the coarsest-level conjugate gradients (k_cg_cluster below).
// Bound by latency (two dependent launches of a few microseconds), in FP64 by the FP64 pipes.  With the
// one-launch CG, V-cycles went from (streaming tiles filling the SMs) 1017 to 703 us (FP32, level 4 / 17
// layers), 3097 to 2772 us (FP32, 6 / 65), 1404 to 1072 us (FP32, two radial points, 5 / 33) and 3999 to 2816 us
// (FP64, 5 / 33).
// Sums run in a fixed order (copies in ascending layout order; corners 00, 10, 01, 11; bottom then top
// contributions), so results do not depend on scheduling.

// Index data of a small level: unique lateral points are the interface groups first, then the points inside
// the diamonds.
struct SmallDims {
  int N, n_r, P, ls, ds, nll;  // ls / ds: layer / diamond stride of the node layout, nll: lateral layout size
  int n_groups, n_lat, ncell;  // interface groups, unique lateral points, cells
  const int* gptr;
  const int64_t* goff;
};
inline SmallDims small_dims(const Level& L) {
  SmallDims s;
  s.N = L.N, s.n_r = L.n_r, s.P = L.P, s.ls = (int)L.layer_stride, s.ds = (int)L.diamond_stride;
  s.nll = (int)L.n_lat_layout;
  s.n_groups = L.n_groups, s.n_lat = 10 * L.N * L.N + 2, s.ncell = 10 * L.N * L.N * (L.n_r - 1);
  s.gptr = L.grp_ptr, s.goff = L.grp_off;
  return s;
}

template <typename T>
struct SmallTab {  // tables of the level in its precision
  const T *geo, *lay, *svec;
  EtaView<T> eta;
  int bc_in, bc_out;
};
template <typename T>
inline SmallTab<T> small_tab(const Level& L, BC bc) {
  return SmallTab<T>{Tab<T>::geo(L), Tab<T>::lay(L), Tab<T>::s(L), etav<T>(L), bc.in, bc.out};
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

// Copies of unique lateral point u: count and, for copy q, (d, i, j).
__device__ __forceinline__ void small_copies(const SmallDims& S, int u, int& b, int& e) {
  if (u < S.n_groups) b = S.gptr[u], e = S.gptr[u + 1];
  else b = 0, e = 1;
}
__device__ __forceinline__ void small_copy(const SmallDims& S, int u, int q, int& d, int& i, int& j) {
  if (u < S.n_groups) {
    const int off = (int)S.goff[q];
    d = off / S.ds;
    const int r = off - d * S.ds;
    i = r / S.P, j = r - i * S.P;
  } else {
    const int w = u - S.n_groups, n1 = S.N - 1, per = n1 * n1;
    d = w / per;
    const int r = w - d * per;
    i = r / n1 + 1, j = r - (i - 1) * n1 + 1;
  }
}

// y = (P A P + I - P) in at unique node (u, k) from the cells' contributions; o0: the layout offset of its
// first copy (the canonical one).
template <typename T, bool CG>
__device__ __forceinline__ void small_node(const SmallDims& S, const SmallTab<T>& B, const T* const (&in)[3],
                                           const T* __restrict__ sc, int u, int k, T (&v)[3], int& o0) {
  int b, e;
  small_copies(S, u, b, e);
  v[0] = v[1] = v[2] = (T)0;
  int lat0 = 0;
  for (int q = b; q < e; ++q) {
    int d, i, j;
    small_copy(S, u, q, d, i, j);
    if (q == b) lat0 = d * S.ls + i * S.P + j, o0 = d * S.ds + k * S.ls + i * S.P + j;
    small_gather(S, sc, d, i, j, k, v);
  }
  if (k == 0 || k == S.n_r - 1) {
    const int bc = k == 0 ? B.bc_in : B.bc_out;
    T w[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) w[x] = CG ? __ldcg(in[x] + o0) : in[x][o0];
    if (bc == TN_BC_NOSLIP) {
#pragma unroll
      for (int x = 0; x < 3; ++x) v[x] = w[x];
    } else {
      const T sx = B.svec[lat0], sy = B.svec[lat0 + S.nll], sz = B.svec[lat0 + 2 * S.nll];
      const T dv = (w[0] - v[0]) * sx + (w[1] - v[1]) * sy + (w[2] - v[2]) * sz;
      v[0] += dv * sx, v[1] += dv * sy, v[2] += dv * sz;
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
  const int t = blockIdx.x * 128 + threadIdx.x;
  if (t >= S.n_lat * S.n_r) return;
  const int k = t / S.n_lat, u = t - k * S.n_lat;
  const T* const in[3] = {in0, in1, in2};
  T v[3];
  int o0;
  small_node<T, false>(S, B, in, sc, u, k, v, o0);
  int b, e;
  small_copies(S, u, b, e);
  for (int q = b; q < e; ++q) {
    const int o = u < S.n_groups ? (int)S.goff[q] + k * S.ls : o0;
    if (EPI != EPI_NONE) {
      epilogue<T, EPI>(E, in0, in1, in2, o, v);
    } else {
      out0[o] = v[0], out1[o] = v[1], out2[o] = v[2];
    }
  }
}

// ---------------------------------------------------------------- coarsest-level conjugate gradients
// The whole block-Jacobi-preconditioned CG of the coarsest level (Sec. 7) in one launch of one cluster of
// eight CTAs: the kernel-per-step form took three launches per step, about 150 in a captured V-cycle, each
// of them a few microseconds of latency for a level of some hundred nodes.  Unique node t = k n_lat + u
// belongs to one thread throughout; its r, z, x live at its canonical layout entry, p at every copy.  Cells
// and nodes go round the CTAs warp by warp; data of other SMs is read past L1 after a cluster
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

template <typename T, typename Op>
__global__ void __launch_bounds__(kCgThreads) k_cg_cluster(SmallDims S, SmallTab<T> B, Op op, CgArgs<T> A) {
  namespace cgr = cooperative_groups;
  cgr::cluster_group cl = cgr::this_cluster();
  __shared__ double wsum[kCgThreads / 32][3], csum[2][kCgCtas][3];
  const int rank = (int)cl.block_rank();
  const int gt = (((int)threadIdx.x >> 5) * kCgCtas + rank) * 32 + ((int)threadIdx.x & 31);
  constexpr int GT = kCgCtas * kCgThreads;
  const int nn = S.n_lat * S.n_r;
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
  auto first = [&](int t, int& o, int& lat, int& k) {  // canonical entry of unique node t
    k = t / S.n_lat;
    const int u = t - k * S.n_lat;
    int b, e, d, i, j;
    small_copies(S, u, b, e);
    small_copy(S, u, b, d, i, j);
    lat = d * S.ls + i * S.P + j, o = lat + d * (S.ds - S.ls) + k * S.ls;
  };
  auto put = [&](int t, const T (&v)[3], T* const (&dst)[3]) {  // to every copy
    const int k = t / S.n_lat, u = t - k * S.n_lat;
    int b, e;
    small_copies(S, u, b, e);
    for (int q = b; q < e; ++q) {
      int d, i, j;
      small_copy(S, u, q, d, i, j);
      const int o = d * S.ds + k * S.ls + i * S.P + j;
#pragma unroll
      for (int c = 0; c < 3; ++c) dst[c][o] = v[c];
    }
  };
  auto bmul3 = [&](int o, const T (&r)[3], T (&z)[3]) {
    const T a = A.binv[0][o], e = A.binv[1][o], f = A.binv[2][o], xy = A.binv[3][o], xz = A.binv[4][o], yz = A.binv[5][o];
    z[0] = a * r[0] + xy * r[1] + xz * r[2];
    z[1] = xy * r[0] + e * r[1] + yz * r[2];
    z[2] = xz * r[0] + yz * r[1] + f * r[2];
  };
  // rotation component: w = Ginv (sum over unique nodes of x cross v), removed as v - w cross x
  auto spin = [&](const T* const (&v)[3], double (&w)[3]) {
    double a[3] = {0, 0, 0};
    for (int t = gt; t < nn; t += GT) {
      int o, lat, k;
      first(t, o, lat, k);
      const double r = A.rad[k];
      const double x[3] = {r * B.svec[lat], r * B.svec[lat + S.nll], r * B.svec[lat + 2 * S.nll]};
      const double y[3] = {v[0][o], v[1][o], v[2][o]};
      a[0] += x[1] * y[2] - x[2] * y[1];
      a[1] += x[2] * y[0] - x[0] * y[2];
      a[2] += x[0] * y[1] - x[1] * y[0];
    }
    total(a, 3);
    for (int c = 0; c < 3; ++c) w[c] = A.ginv[3 * c] * a[0] + A.ginv[3 * c + 1] * a[1] + A.ginv[3 * c + 2] * a[2];
  };
  auto despin = [&](int lat, int k, const double (&w)[3], T (&v)[3]) {
    const double r = A.rad[k];
    const double x[3] = {r * B.svec[lat], r * B.svec[lat + S.nll], r * B.svec[lat + 2 * S.nll]};
    v[0] -= (T)(w[1] * x[2] - w[2] * x[1]);
    v[1] -= (T)(w[2] * x[0] - w[0] * x[2]);
    v[2] -= (T)(w[0] * x[1] - w[1] * x[0]);
  };

  double w[3] = {0, 0, 0}, acc[3];
  const T* const bb[3] = {A.b0, A.b1, A.b2};
  if (A.project) spin(bb, w);
  // r = b (rotations removed), z = D^-1 r, p = z, x = 0
  acc[0] = 0.0;
  for (int t = gt; t < nn; t += GT) {
    int o, lat, k;
    first(t, o, lat, k);
    T r[3] = {A.b0[o], A.b1[o], A.b2[o]}, z[3];
    if (A.project) despin(lat, k, w, r);
    bmul3(o, r, z);
    T d = (T)0;
#pragma unroll
    for (int c = 0; c < 3; ++c) A.r[c][o] = r[c], A.x[c][o] = (T)0, d += r[c] * z[c];
    acc[0] += (double)d;
    put(t, z, A.p);
  }
  total(acc, 1);
  const double rz0 = acc[0];
  double rz = rz0;
  const T* const pp[3] = {A.p[0], A.p[1], A.p[2]};
  if (rz0 > 0.0) {
    for (int it = 0; it < A.maxit; ++it) {
      for (int c = gt; c < S.ncell; c += GT) small_cell<T, Op, true>(S, B, op, pp, c, A.sc);
      cl.sync();
      // q = K p, kept in z until the update
      acc[0] = 0.0;
      for (int t = gt; t < nn; t += GT) {
        T q[3];
        int o;
        small_node<T, true>(S, B, pp, A.sc, t % S.n_lat, t / S.n_lat, q, o);
        T d = (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) A.z[c][o] = q[c], d += A.p[c][o] * q[c];
        acc[0] += (double)d;
      }
      total(acc, 1);
      const T al = (T)(rz / acc[0]);
      acc[0] = 0.0;
      for (int t = gt; t < nn; t += GT) {
        int o, lat, k;
        first(t, o, lat, k);
        T r[3], z[3], d = (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          A.x[c][o] += al * A.p[c][o];
          r[c] = A.r[c][o] - al * A.z[c][o];
          A.r[c][o] = r[c];
        }
        bmul3(o, r, z);
#pragma unroll
        for (int c = 0; c < 3; ++c) A.z[c][o] = z[c], d += r[c] * z[c];
        acc[0] += (double)d;
      }
      total(acc, 1);
      const double rzn = acc[0];
      if (!(rzn > A.tol2 * rz0) || it == A.maxit - 1) break;
      const T be = (T)(rzn / rz);
      rz = rzn;
      for (int t = gt; t < nn; t += GT) {
        int o, lat, k;
        first(t, o, lat, k);
        T p[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) p[c] = A.z[c][o] + be * A.p[c][o];
        put(t, p, A.p);
      }
      cl.sync();
    }
  }
  // x (rotations removed) to every copy
  const T* const xx[3] = {A.x[0], A.x[1], A.x[2]};
  if (A.project) spin(xx, w);
  for (int t = gt; t < nn; t += GT) {
    int o, lat, k;
    first(t, o, lat, k);
    T x[3] = {A.x[0][o], A.x[1][o], A.x[2][o]};
    if (A.project) despin(lat, k, w, x);
    put(t, x, A.x);
  }
  cl.sync();  // no CTA leaves while another may still write its shared memory
}
