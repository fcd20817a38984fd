// Divergence B and gradient B^T with the pressure transfers inside (included by kernels.cu inside its
// namespace).  The pressure lives one level coarser, so B is the element divergence followed by the transposed
// interpolation and B^T the interpolation followed by the element gradient; both run here in one kernel over
// coarse cell layers (two fine cell layers at a time), with no fine-level intermediate in memory.
//
// Measured (B + B^T with their interface passes): level 7 / 129 layers FP64 3.76 -> 1.93 ms, 6 / 65 FP32 186 -> 98 us,
// 5 / 101 FP64 278 -> 162 us.
//
// Compute type C: float, double, or double-float on FP64 levels with N >= 32 (unnormalised running sums, see
// acc2 in dfloat.cuh).  All arithmetic is on pairs of C: Pr<C>.
template <typename C>
struct Pr;
template <>
struct Pr<float> {
  using V = float2;
  static __device__ __forceinline__ V mk(float a, float b) { return make_float2(a, b); }
  static __device__ __forceinline__ float x(V a) { return a.x; }
  static __device__ __forceinline__ float y(V a) { return a.y; }
  static __device__ __forceinline__ V add(V a, V b) { return add2(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return sub2(a, b); }
  static __device__ __forceinline__ V mul(V a, V b) { return mul2(a, b); }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return fma2(a, b, c); }
  static __device__ __forceinline__ V half(V a) { return mul2(a, make_float2(0.5f, 0.5f)); }
  static __device__ __forceinline__ V norm(V a) { return a; }
  static __device__ __forceinline__ V add_half(V s, V a) { return fma2(a, make_float2(0.5f, 0.5f), s); }
  static __device__ __forceinline__ V add_3half(V s, V a) { return fma2(a, make_float2(1.5f, 1.5f), s); }
  // node sums of the divergence, compensated (TwoSum: s + e is the sum up to the rounding of e)
  static __device__ __forceinline__ void acc(V& s, V& e, V x) {
    const V t = add2(s, x), b = sub2(t, s);
    e = add2(e, add2(sub2(s, sub2(t, b)), sub2(x, b)));
    s = t;
  }
  static __device__ __forceinline__ V close(V s, V e) {  // (an infinite sum has no rounding error: e is not a number then)
    const V t = add2(s, e);
    return make_float2(t.x == t.x ? t.x : s.x, t.y == t.y ? t.y : s.y);
  }
  static __device__ __forceinline__ float in(float v) { return v; }
  template <typename T>
  static __device__ __forceinline__ T out(float v) { return v; }
};
template <>
struct Pr<double> {
  using V = double2;
  static __device__ __forceinline__ V mk(double a, double b) { return make_double2(a, b); }
  static __device__ __forceinline__ double x(V a) { return a.x; }
  static __device__ __forceinline__ double y(V a) { return a.y; }
  static __device__ __forceinline__ V add(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ V sub(V a, V b) { return make_double2(a.x - b.x, a.y - b.y); }
  static __device__ __forceinline__ V mul(V a, V b) { return make_double2(a.x * b.x, a.y * b.y); }
  static __device__ __forceinline__ V fma(V a, V b, V c) {
    return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
  }
  static __device__ __forceinline__ V half(V a) { return make_double2(0.5 * a.x, 0.5 * a.y); }
  static __device__ __forceinline__ V norm(V a) { return a; }
  static __device__ __forceinline__ V add_half(V s, V a) { return fma(a, make_double2(0.5, 0.5), s); }
  static __device__ __forceinline__ V add_3half(V s, V a) { return fma(a, make_double2(1.5, 1.5), s); }
  static __device__ __forceinline__ void acc(V& s, V&, V x) { s = add(s, x); }
  static __device__ __forceinline__ V close(V s, V) { return s; }
  static __device__ __forceinline__ double in(double v) { return v; }
  template <typename T>
  static __device__ __forceinline__ T out(double v) { return v; }
};
template <>
struct Pr<dfl> {
  using V = df2;
  static __device__ __forceinline__ V mk(const dfl& a, const dfl& b) { return pack(a, b); }
  static __device__ __forceinline__ dfl x(const V& a) { return lane_x(a); }
  static __device__ __forceinline__ dfl y(const V& a) { return lane_y(a); }
  static __device__ __forceinline__ V add(const V& a, const V& b) { return df_of(sum2(a, b)); }
  static __device__ __forceinline__ V sub(const V& a, const V& b) { return diff2(a, b); }
  static __device__ __forceinline__ V mul(const V& a, const V& b) { return df_of(prod2(a, b)); }
  static __device__ __forceinline__ V fma(const V& a, const V& b, const V& c) {
    acc2 s = acc_of(c);
    acc_fma2(s, a, b);
    return df_of(s);
  }
  static __device__ __forceinline__ V half(const V& a) {
    const float2 h = make_float2(0.5f, 0.5f);
    return df2{p2mul(a.hi, h), p2mul(a.lo, h)};
  }
  static __device__ __forceinline__ V norm(const V& a) { return norm2(a); }
  static __device__ __forceinline__ V add_half(const V& s, const V& a) { return add(s, half(a)); }
  static __device__ __forceinline__ V add_3half(const V& s, const V& a) { return add(s, add(a, half(a))); }
  static __device__ __forceinline__ void acc(V& s, V&, const V& x) { s = add(s, x); }
  static __device__ __forceinline__ const V& close(const V& s, const V&) { return s; }
  static __device__ __forceinline__ dfl in(double v) { return split(v); }
  template <typename T>
  static __device__ __forceinline__ T out(const dfl& v) { return join(v); }
};

// The six triangles around node (i, j): cell offset, wedge, the node's local index, and the triangle's two
// other nodes among the neighbours 1 .. 6 = (1,0) (0,1) (-1,1) (-1,0) (0,-1) (1,-1) (0 is the node itself).
__device__ constexpr int kTri[6][6] = {{0, 0, 0, 0, 1, 2},  {-1, 0, 1, 2, 2, 3},  {-1, 0, 0, 1, 3, 4},
                                       {-1, -1, 1, 0, 4, 5}, {0, -1, 0, 2, 5, 6}, {0, -1, 1, 1, 6, 1}};

// ------------------------------------------------------------------------------------ gradient
// y_n = sum over the triangles t around n of g_a(t) A_t + m(t) G_t with g_a = |det M| l_a, m = |det M| m2 (rows
// of M^-1, l_0 = -(m0 + m1), l_1 = m0, l_2 = m1) and A_t, G_t the sums over t's nodes of the radial
// combinations at node layer k
//   alpha = a_k + a_k-1,  gamma = r_k-1 a_k-1 - r_k a_k,  a_k = -vol w0 / 6 (p_k + p_k+1),
// so a node is a seven-point stencil of (alpha, gamma) with weights that do not depend on the layer: 21 pair
// products per node and layer, no exchange of contributions.  One thread per node of a 16 x 16 tile keeps its
// weights in shared memory; the nodes of the tile and of a one-node rim form (alpha, gamma) of two layers from
// the coarse pressure.  The diamond's last row and column (i = N, j = N) are strips of their own.
// Bound by the FP32 pipe (double-float: 42 x 10 packed operations per node and coarse layer) or by memory.
constexpr int kGrTile = 16, kGrThreads = 256, kGrStrip = 128, kGrRim = 400;  // rim: 18 x 18 and 3 x 130 nodes
constexpr int kGrMaxKc = 64;                                                 // coarse cell layers per chunk at most
template <typename C>
constexpr size_t grad_smem_bytes() {
  return sizeof(typename Pr<C>::V) * (size_t)((sizeof(C) == 4 ? 0 : 21 * kGrThreads) + 4 * kGrRim + 2 * (kGrMaxKc + 1));
}

template <typename T, typename C>
__global__ void __launch_bounds__(kGrThreads, 2)
    k_grad(Dims F, Dims Cc, int ntile, const T* __restrict__ p, T* __restrict__ y0, T* __restrict__ y1,
           T* __restrict__ y2, const T* __restrict__ geo, const C* __restrict__ lay, const T* __restrict__ svec,
           int bc_in, int bc_out, int kc) {
  using R = Pr<C>;
  using V = typename R::V;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  constexpr bool WREG = sizeof(C) == 4;  // FP32 weights stay in registers
  V* const wt = reinterpret_cast<V*>(tile_smem) + threadIdx.x;                        // [7][3][kGrThreads] (g, m)
  V* const ag = reinterpret_cast<V*>(tile_smem) + (WREG ? 0 : 21 * kGrThreads);       // [2][2][kGrRim] (alpha, gamma)
  V* const lct = ag + 4 * kGrRim;                                                     // [kGrMaxKc + 1][2]
  V wr[WREG ? 21 : 1];
  const int N = F.N, n_r = F.n_r, P = F.P, LS = (int)F.layer_stride;
  const int d = blockIdx.z, nK = (n_r - 1) / 2;
  // this CTA's nodes: rows i0 .. i0 + TI - 1, columns j0 .. j0 + TJ - 1
  int i0, j0, TI, TJ;
  {
    const int nt = N / ntile, main = nt * nt, rows = (N + kGrStrip) / kGrStrip, b = blockIdx.x;
    if (b < main) i0 = (b / nt) * ntile, j0 = (b % nt) * ntile, TI = TJ = ntile;
    else if (b < main + rows) i0 = N, TI = 1, j0 = (b - main) * kGrStrip, TJ = min(kGrStrip, N + 1 - j0);
    else j0 = N, TJ = 1, i0 = (b - main - rows) * kGrStrip, TI = min(kGrStrip, N - i0);
  }
  const int t = threadIdx.x, ti = t / TJ, tj = t - ti * TJ;
  const bool own = ti < TI;
  const int i = i0 + ti, j = j0 + tj;
  // weights of this thread's node
  if (own) {
    V w[7][3];
    const V zero = R::mk(C(0.0f), C(0.0f));
#pragma unroll
    for (int n = 0; n < 7; ++n) w[n][0] = w[n][1] = w[n][2] = zero;
    const int nt = (int)F.n_tri;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int ci = i + kTri[q][0], cj = j + kTri[q][1];
      if (ci < 0 || cj < 0 || ci >= N || cj >= N) continue;
      const int tr = ((d * N + ci) * N + cj) * 2 + kTri[q][2];
      const C dm = R::in(geo[9 * nt + tr]);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const C m2 = R::in(geo[(6 + c) * nt + tr]);
        V l;
        if (kTri[q][3] == 0) {  // (-(m0 + m1), m2)
          const C a = R::in(geo[c * nt + tr]), b = R::in(geo[(3 + c) * nt + tr]);
          l = R::sub(R::mk(-a, m2), R::mk(b, C(0.0f)));
        } else {
          l = R::mk(R::in(geo[(kTri[q][3] == 1 ? c : 3 + c) * nt + tr]), m2);
        }
        w[0][c] = R::fma(R::mk(dm, dm), l, w[0][c]);
        w[kTri[q][4]][c] = R::fma(R::mk(dm, dm), l, w[kTri[q][4]][c]);
        w[kTri[q][5]][c] = R::fma(R::mk(dm, dm), l, w[kTri[q][5]][c]);
      }
    }
#pragma unroll
    for (int n = 0; n < 7; ++n)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if constexpr (WREG) wr[3 * n + c] = w[n][c];
        else wt[(3 * n + c) * kGrThreads] = R::norm(w[n][c]);
      }
  }
  // rim nodes e = t, t + 256: offsets of their two coarse lateral parents (equal for a coarse node)
  const int W = TJ + 2, H = (TI + 2) * W;  // <= 390
  int off0[2], off1[2];
  bool on[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int e = t + s * kGrThreads, hi = i0 - 1 + e / W, hj = j0 - 1 + e % W;
    on[s] = e < H && hi >= 0 && hj >= 0 && hi <= N && hj <= N;
    const int oi = hi & 1, oj = hj & 1;
    const int I0 = (hi + oi * (2 * oj - 1)) >> 1, J0 = (hj - oj) >> 1, I1 = (hi + oi * (1 - 2 * oj)) >> 1, J1 = (hj + oj) >> 1;
    const int b = (int)(d * Cc.diamond_stride);
    off0[s] = b + I0 * Cc.P + J0, off1[s] = b + I1 * Cc.P + J1;
    if (!on[s] && e < H)
#pragma unroll
      for (int q = 0; q < 4; ++q) ag[q * kGrRim + e] = R::mk(C(0.0f), C(0.0f));
  }
  const int CLS = (int)Cc.layer_stride;
  const int K0 = blockIdx.y * kc, K1 = min(nK, K0 + kc), Kb = max(K0 - 1, 0);
  for (int K = Kb + t; K < K1; K += kGrThreads) {  // (-vol w0 / 6, r) of the fine cell layers 2K, 2K + 1
    const C *l0 = lay + kLayerStride * (2 * K), *l1 = l0 + kLayerStride;
    lct[2 * (K - Kb)] = R::mk(l0[7], l1[7]), lct[2 * (K - Kb) + 1] = R::mk(l0[4], l1[4]);
  }
  __syncthreads();
  T raw0[2], raw1[2];
  auto request = [&](int K) {
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (on[s]) raw0[s] = p[off0[s] + K * CLS], raw1[s] = p[off1[s] + K * CLS];
  };
  auto lateral = [&](int s) {  // pressure at the rim node's lateral position on a coarse layer
    return R::x(R::half(R::add(R::mk(R::in(raw0[s]), R::in(raw0[s])), R::mk(R::in(raw1[s]), R::in(raw1[s])))));
  };
  // P_2K = S + L_K, P_2K+1 = S + L_K+1 with S = (L_K + L_K+1) / 2; a, b = r a of both fine cell layers
  auto cell_pair = [&](int K, const C& lo, const C& hi, V& f, V& r, V& P, V& a, V& b) {
    const V S = R::half(R::add(R::mk(lo, lo), R::mk(hi, hi)));
    f = lct[2 * (K - Kb)], r = lct[2 * (K - Kb) + 1];
    P = R::add(S, R::mk(lo, hi)), a = R::mul(f, P), b = R::mul(r, a);
  };
  C L[2], ap[2], bp[2];  // coarse-layer value, a and b of the cell layer below
#pragma unroll
  for (int s = 0; s < 2; ++s) L[s] = ap[s] = bp[s] = C(0.0f), raw0[s] = raw1[s] = (T)0;
  if (K0 > 0) {
    C lo[2];
    request(K0 - 1);
#pragma unroll
    for (int s = 0; s < 2; ++s) lo[s] = lateral(s);
    request(K0);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      L[s] = lateral(s);
      V f, r, P, a, b;
      cell_pair(K0 - 1, lo[s], L[s], f, r, P, a, b);
      ap[s] = R::y(a), bp[s] = R::y(b);
    }
  } else {
    request(0);
#pragma unroll
    for (int s = 0; s < 2; ++s) L[s] = lateral(s);
  }
  const int nd = (ti + 1) * W + tj + 1;
  const int nb[7] = {nd, nd + W, nd + 1, nd - W + 1, nd - W, nd - 1, nd + W - 1};
  const int o0 = (int)(d * F.diamond_stride) + i * P + j;
  const int64_t so = (int64_t)d * (N + 1) * P + i * P + j;
  auto emit = [&](const V (&acc)[3], int k) {
    T o[3];
    const V z01 = R::add(R::mk(R::x(acc[0]), R::x(acc[1])), R::mk(R::y(acc[0]), R::y(acc[1])));
    const V z2 = R::add(acc[2], R::mk(R::y(acc[2]), R::x(acc[2])));
    o[0] = R::template out<T>(R::x(z01)), o[1] = R::template out<T>(R::y(z01)), o[2] = R::template out<T>(R::x(z2));
    if (k == 0 || k == n_r - 1) project_vec(o, svec, so, F.n_lat_layout, k == 0 ? bc_in : bc_out);
    const int o_ = o0 + k * LS;
    y0[o_] = o[0], y1[o_] = o[1], y2[o_] = o[2];
  };
  auto nodes = [&](const V* v, int k, bool two) {  // the stencil at node layer k, and k + 1 from the next half
    V a0[3], a1[3];
#pragma unroll
    for (int n = 0; n < 7; ++n) {
      const V x0 = v[nb[n]], x1 = v[kGrRim + nb[n]];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        V w;
        if constexpr (WREG) w = wr[3 * n + c];
        else w = wt[(3 * n + c) * kGrThreads];
        a0[c] = n == 0 ? R::mul(w, x0) : R::fma(w, x0, a0[c]);
        a1[c] = n == 0 ? R::mul(w, x1) : R::fma(w, x1, a1[c]);
      }
    }
    emit(a0, k);
    if (two) emit(a1, k + 1);
  };
  request(K0 + 1);
  for (int K = K0; K < K1; ++K) {
    V* const buf = ag + (K & 1) * 2 * kGrRim;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!on[s]) continue;
      const C hi = lateral(s);
      V f, r, P, a, b;
      cell_pair(K, L[s], hi, f, r, P, a, b);
      // alpha = f P + the layer below's a, gamma = the layer below's b - r a
      const V al = R::norm(R::fma(f, P, R::mk(ap[s], R::x(a))));
      const V ga = R::norm(R::fma(R::mk(-R::x(r), -R::y(r)), a, R::mk(bp[s], R::x(b))));
      const int e = t + s * kGrThreads;
      buf[e] = R::mk(R::x(al), R::x(ga)), buf[kGrRim + e] = R::mk(R::y(al), R::y(ga));
      L[s] = hi, ap[s] = R::y(a), bp[s] = R::y(b);
    }
    if (K + 2 <= K1) request(K + 2);
    // a buffer is rewritten two coarse layers later, past the next barrier, which follows its reads
    __syncthreads();
    if (own) nodes(buf, 2 * K, true);
  }
  if (K1 == nK) {  // the top node layer: contributions of the last cell layer only
    V* const buf = ag + (K1 & 1) * 2 * kGrRim;
#pragma unroll
    for (int s = 0; s < 2; ++s)
      if (on[s]) buf[t + s * kGrThreads] = buf[kGrRim + t + s * kGrThreads] = R::mk(ap[s], bp[s]);
    __syncthreads();
    if (own) nodes(buf, n_r - 1, false);
  }
}

// ------------------------------------------------------------------------------------ divergence
// With Lam_t,k = sum over a of u_a,k . l_a on node layer k and Mu_t,k = (sum over a of u_a,k+1 - u_a,k) . m2, wedge (t, k)
// has
//   v_t,k = -vol w0 |det M| / 6 (Lam_k + Lam_k+1 + r_k Mu_k),
// differences of nodal values before any product: r grows with the number of layers, and a rounded
// (sum over a of u_a,k) . m2 per node layer, differenced afterwards, loses as many digits on smooth velocities
// (error in norm over the interior nodes, sines and polynomials at level 5 / 101 layers: FP32 1.9e-7 that way,
// 6.0e-8 this way; double-float 4.0e-14 and 9.6e-15; FP32 saddle 6 / 65 93 -> 98 us, FP64 5 / 101 158 -> 162 us).
// The coarse pressure node (I, J, K) sums 6 psi(q_c) v: laterally 2, 1/2, 1/2 (the coarse triangle's corner
// child at the node, the other two) and 1 (the middle child), radially 1/2, 3/2, 3/2, 1/2 over the fine cell
// layers 2K - 2 .. 2K + 1.  A CTA owns ntile / 2 x ntile / 2 coarse nodes, one thread per fine cell of the tile
// and of a rim of two cells at its low edges; Lam is formed once per node layer and Mu once per cell layer, from a ring
// of three node layers in shared memory (of which a coarse layer replaces two), and the lateral
// sums run once per coarse layer: within a coarse cell first (four threads, one corner each), then over the
// coarse cells around a node.  Bound by the FP32 pipe (double-float) or by memory.
constexpr int kDvTile = 16, kDvThreads = 352, kDvCells = (kDvTile + 2) * (kDvTile + 2),
              kDvNodes = (kDvTile + 3) * (kDvTile + 3), kDvMaxKc = 32;
template <typename T, typename C>
constexpr size_t div_smem_bytes() {
  return sizeof(typename Pr<C>::V) * (size_t)(13 * kDvCells + 2 * (kDvMaxKc + 1)) +
         (3 * sizeof(C) + 2 * sizeof(T)) * (size_t)(3 * kDvNodes);
}
static_assert(div_smem_bytes<double, dfl>() <= 113 * 1024, "two CTAs per SM");
__device__ __forceinline__ void cp_async_elem(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_elem(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

template <typename T, typename C>
__global__ void __launch_bounds__(kDvThreads, 2)
    k_div(Dims F, Dims Cc, int ntile, const T* __restrict__ in0, const T* __restrict__ in1, const T* __restrict__ in2,
          T* __restrict__ q, const T* __restrict__ geo, const C* __restrict__ lay, const T* __restrict__ svec,
          int bc_in, int bc_out, int kc) {
  using R = Pr<C>;
  using V = typename R::V;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  V* const gc = reinterpret_cast<V*>(tile_smem) + threadIdx.x;    // [10][kDvCells] M^-1, |det M|
  V* const tb = reinterpret_cast<V*>(tile_smem) + 10 * kDvCells;  // [2][kDvCells] (bottom, top) of W0, W1
  V* const cb = tb + 2 * kDvCells;                                // [kDvCells] of coarse-cell corners
  V* const lct = cb + kDvCells;                                   // [kDvMaxKc + 1][2]
  C* const us = reinterpret_cast<C*>(lct + 2 * (kDvMaxKc + 1));   // [3][3][kDvNodes]: ring of three node layers
  T* const rw = reinterpret_cast<T*>(us + 3 * 3 * kDvNodes);      // [2][3][kDvNodes]: the next two, as stored
  const int N = F.N, n_r = F.n_r, P = F.P, LS = (int)F.layer_stride;
  const int d = blockIdx.z, nK = (n_r - 1) / 2;
  const int nt_ = N / ntile, W = ntile + 2, WN = ntile + 3;
  const int i0 = ((int)blockIdx.x / nt_) * ntile - 2, j0 = ((int)blockIdx.x % nt_) * ntile - 2;  // first cell
  const int t = threadIdx.x, ti = t / W, tj = t - ti * W;
  const int ci = i0 + ti, cj = j0 + tj;
  const bool in_tile = ti < W, cell = in_tile && ci >= 0 && cj >= 0;
  const int dbase = (int)(d * F.diamond_stride), lbase = d * (N + 1) * P;
  // node loads: own node (corner 00 of the cell), and the far row and column by threads 0 .. 2 WN - 2
  const int slot = ti * WN + tj;
  int xs = -1, xi = 0, xj = 0;
  if (t < 2 * WN - 1) {
    const int si = t < WN ? W : t - WN, sj = t < WN ? t : W;
    xi = i0 + si, xj = j0 + sj;
    if (xi >= 0 && xj >= 0) xs = si * WN + sj;
  }
  const int c00 = dbase + ci * P + cj, x00 = dbase + xi * P + xj;
  const int K0 = blockIdx.y * kc, K1 = min(nK, K0 + kc), Kb = max(K0 - 1, 0);  // coarse cell layers Kb .. K1 - 1
  // request of this thread's nodes on layers k, k + 1 (read back by the thread itself)
  auto request = [&](int k) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T* const r = rw + h * 3 * kDvNodes;
      if (cell) {
        const int o = c00 + (k + h) * LS;
        cp_async_elem(smem_u32(r + slot), in0 + o), cp_async_elem(smem_u32(r + kDvNodes + slot), in1 + o);
        cp_async_elem(smem_u32(r + 2 * kDvNodes + slot), in2 + o);
      }
      if (xs >= 0) {
        const int o = x00 + (k + h) * LS;
        cp_async_elem(smem_u32(r + xs), in0 + o), cp_async_elem(smem_u32(r + kDvNodes + xs), in1 + o);
        cp_async_elem(smem_u32(r + 2 * kDvNodes + xs), in2 + o);
      }
    }
    cp_async_commit();
  };
  auto put = [&](int k, int h, T (&v)[3], int s, int64_t so) {  // projected on the boundary layers
    if (k == 0 || k == n_r - 1) project_vec(v, svec, so, F.n_lat_layout, k == 0 ? bc_in : bc_out);
#pragma unroll
    for (int c = 0; c < 3; ++c) us[h + c * kDvNodes + s] = R::in(v[c]);
  };
  auto put2 = [&](int k, int h1, int h2) {  // the requested layers k, k + 1
    cp_async_wait<0>();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const T* const r = rw + h * 3 * kDvNodes;
      if (cell) {
        T v[3] = {r[slot], r[kDvNodes + slot], r[2 * kDvNodes + slot]};
        put(k + h, h == 0 ? h1 : h2, v, slot, (int64_t)lbase + ci * P + cj);
      }
      if (xs >= 0) {
        T v[3] = {r[xs], r[kDvNodes + xs], r[2 * kDvNodes + xs]};
        put(k + h, h == 0 ? h1 : h2, v, xs, (int64_t)lbase + xi * P + xj);
      }
    }
  };
  {  // the first node layer
    T v[3];
    if (cell) {
      const int o = c00 + 2 * Kb * LS;
      v[0] = in0[o], v[1] = in1[o], v[2] = in2[o];
      put(2 * Kb, 0, v, slot, (int64_t)lbase + ci * P + cj);
    }
    if (xs >= 0) {
      const int o = x00 + 2 * Kb * LS;
      v[0] = in0[o], v[1] = in1[o], v[2] = in2[o];
      put(2 * Kb, 0, v, xs, (int64_t)lbase + xi * P + xj);
    }
  }
  request(2 * Kb + 1);
  if (cell) {
    const int t0 = ((d * N + ci) * N + cj) * 2, nt = (int)F.n_tri;
#pragma unroll
    for (int g = 0; g < 10; ++g) gc[g * kDvCells] = R::mk(R::in(geo[g * nt + t0]), R::in(geo[g * nt + t0 + 1]));
  }
  for (int K = Kb + t; K < K1; K += kDvThreads) {  // (-vol w0 / 6, r) of the fine cell layers 2K, 2K + 1
    const C *l0 = lay + kLayerStride * (2 * K), *l1 = l0 + kLayerStride;
    lct[2 * (K - Kb)] = R::mk(l0[7], l0[4]), lct[2 * (K - Kb) + 1] = R::mk(l1[7], l1[4]);
  }
  const V zero = R::mk(C(0.0f), C(0.0f));
  if (in_tile && !cell) tb[t] = tb[kDvCells + t] = zero;  // cells outside the diamond
  auto corners = [&](int h, V& a, V& b) {  // u at the corners (00, 11) and (10, 01), from offset h of us
    const C* const u = us + h;
    a = R::mk(u[0], u[WN + 1]), b = R::mk(u[WN], u[1]);
  };
  auto lateral = [&](int c, const V& a, const V& b, V& lam) {  // + component c of Lam, a and b its corners
    // (differences normalised: after a cancellation their low part is large, and the products drop low x low)
    const V ax = R::norm(R::sub(b, a)), ay = R::norm(R::sub(R::mk(R::y(b), R::x(b)), a));
    lam = c == 0 ? R::mul(ax, gc[0]) : R::fma(ax, gc[c * kDvCells], lam);
    lam = R::fma(ay, gc[(3 + c) * kDvCells], lam);
  };
  auto radial = [&](int c, const V& a0, const V& b0, const V& a1, const V& b1, V& mu) {  // + component c of Mu
    const V da = R::sub(a1, a0), db = R::sub(b1, b0);
    const V dz = R::norm(R::add(R::add(db, R::mk(R::y(db), R::x(db))), da));
    mu = c == 0 ? R::mul(dz, gc[6 * kDvCells]) : R::fma(dz, gc[(6 + c) * kDvCells], mu);
  };
  auto wedge = [&](const V& fr, const V& lam0, const V& lam1, const V& mu) {
    const V f = R::mul(R::mk(R::x(fr), R::x(fr)), gc[9 * kDvCells]);
    return R::mul(f, R::fma(R::mk(R::y(fr), R::y(fr)), mu, R::add(lam0, lam1)));
  };
  // coarse corner of this thread's coarse cell (four threads per coarse cell): q = 2 * (tj & 1) + (ti & 1)
  const int bt = (ti & ~1) * W + (tj & ~1);  // fine cell (2I, 2J) of the coarse cell
  const int corner = (ti & 1) + 2 * (tj & 1);
  // coarse nodes of the tile, one thread each; the last tiles also own I = N / 2, J = N / 2.  FP32: by the last warps, which
  // hold the fewest cells (repeated saddle passes at 6 / 65 94.5 -> 92.8 us); the others by the first (double-float 5 / 101 156.6 against 158 us)
  const int ho = ntile / 2, ni = ho + (i0 + 2 + ntile == N), nj = ho + (j0 + 2 + ntile == N);
  const int ot = t - (sizeof(C) == 4 ? kDvThreads - 96 : 0);
  const bool owner = ot >= 0 && ot < ni * nj;
  const int oi = ot / nj, oj = ot - oi * nj;  // coarse cell row / column oi + 1 of the tile has the node as corner 00
  const int qo = (int)(d * Cc.diamond_stride) + ((i0 + 2) / 2 + oi) * Cc.P + (j0 + 2) / 2 + oj;
  // FP32 sums compensated: the values around a node cancel (wedges that share a node layer enter with opposite signs)
  C carry = C(0.0f), ecarry = C(0.0f);
  auto finish = [&](int K) {  // coarse node layer K from the corners of coarse cell layer K (and the carried ones)
    const V* const c = cb;
    // coarse cells (oi + 1, oj + 1) corner 00, (oi, oj + 1) corner 10, (oi + 1, oj) corner 01, (oi, oj) corner 11 of
    // the tile, those inside it (the far edge's nodes have no cell beyond)
    V s = zero, e = zero;
    const int r1 = 2 * (oi + 1) * W, r0 = 2 * oi * W, c1 = 2 * (oj + 1), c0 = 2 * oj;
    if (oi < ho && oj < ho) s = c[r1 + c1];
    if (oj < ho) R::acc(s, e, c[r0 + W + c1]);
    if (oi < ho) R::acc(s, e, c[r1 + c0 + 1]);
    R::acc(s, e, c[r0 + W + c0 + 1]);
    if (K >= K0) {
      V z = R::mk(R::x(s), R::x(s)), ez = R::mk(R::x(e), R::x(e));
      R::acc(z, ez, R::mk(carry, carry));
      ez = R::add(ez, R::mk(ecarry, ecarry));
      q[qo + K * (int)Cc.layer_stride] = R::template out<T>(R::x(R::close(z, ez)));
    }
    carry = R::y(s), ecarry = R::y(e);
  };
  V lam = zero;
  int h0 = 0, h1 = 3 * kDvNodes, h2 = 2 * 3 * kDvNodes;  // node layers 2K, 2K + 1, 2K + 2 in us
  __syncthreads();
  if (cell)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      V a, b;
      corners(h0 + c * kDvNodes + slot, a, b);
      lateral(c, a, b, lam);
    }
  for (int K = Kb; K < K1; ++K) {
    // (h1, h2 held the layers 2K - 2 and 2K - 1, last read before the previous barrier)
    put2(2 * K + 1, h1, h2);
    if (K + 1 < K1) request(2 * K + 3);
    __syncthreads();
    if (K > Kb && owner) finish(K - 1);
    if (cell) {
      V l1, l2, m1, m2;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        V a0, b0, a1, b1;
        corners(h0 + c * kDvNodes + slot, a0, b0), corners(h1 + c * kDvNodes + slot, a1, b1);
        radial(c, a0, b0, a1, b1, m1);
        corners(h2 + c * kDvNodes + slot, a0, b0);
        radial(c, a1, b1, a0, b0, m2);
        lateral(c, a1, b1, l1), lateral(c, a0, b0, l2);
      }
      const V v0 = wedge(lct[2 * (K - Kb)], lam, l1, m1), v1 = wedge(lct[2 * (K - Kb) + 1], l1, l2, m2);
      lam = l2;
      const V b = R::add_3half(R::half(v1), v0), tp = R::add_3half(R::half(v0), v1);
      tb[t] = R::mk(R::x(b), R::x(tp)), tb[kDvCells + t] = R::mk(R::y(b), R::y(tp));
    }
    __syncthreads();
    if (in_tile) {
      // children of the coarse cell: W0 = (W0 at 00, 10, 01; W1 at 00), W1 = (W1 at 11, 01, 10; W0 at 11); a node
      // gets the middle child + (corner children) / 2 + 3/2 of the corner child at the node
      const V *w0 = tb + bt, *w1 = tb + kDvCells + bt;
      const V a0 = w0[0], a1 = w0[W], a2 = w0[1], am = w1[0], b0 = w1[W + 1], b1 = w1[1], b2 = w1[W], bm = w0[W + 1];
      V r = zero;
      if (corner != 3) r = R::add_3half(R::add_half(am, R::add(R::add(a0, a1), a2)), corner == 0 ? a0 : corner == 1 ? a1 : a2);
      if (corner != 0) {
        const V s = R::add_3half(R::add_half(bm, R::add(R::add(b0, b1), b2)), corner == 3 ? b0 : corner == 1 ? b2 : b1);
        r = corner == 3 ? s : R::add(r, s);
      }
      cb[t] = r;
    }
    // cb is read between the next two barriers and rewritten after them, tb after the next one
    const int h = h0;
    h0 = h2, h2 = h1, h1 = h;
  }
  __syncthreads();
  if (owner) {
    finish(K1 - 1);
    if (K1 == nK) q[qo + nK * (int)Cc.layer_stride] = R::template out<T>(R::x(R::close(R::mk(carry, carry), R::mk(ecarry, ecarry))));
  }
}
