// Double-float A apply of FP64 levels with N >= 32 (included by kernels.cu inside its namespace, after the
// halo-free tiles, whose ring buffer and tile-line pass it shares).
//
// Bound by the FP32 pipe: its rate in lane operations is the same packed or scalar (37.7 and 36.8 T lane-ops/s
// measured), but packed and scalar instructions in turn reach only 29 T, so everything runs packed -- the two
// wedges of a cell in the lanes of the element arithmetic, sums and differences of a node (s, d) and the
// lateral sums of its contributions (X, Y) in the lanes of the node arithmetic.  What it saves against
// k_tile_hf<OpA<dfl>>:
//   * contractions as unnormalised running sums (acc2, dfloat.cuh): 24 packed operations per three products
//     instead of 39;
//   * the four cells around a node are summed laterally before the radial combination.  A cell gives a node
//     X -/+ Y (bottom / top), so a node needs two four-term sums and three additions per component instead of
//     the 15 additions of summing bottom and top contributions apart; only the node's own X + Y is carried to
//     the next layer (6 registers instead of 24);
//   * one barrier per layer: the exchange arrays of consecutive layers alternate, and the nodes of layer k are
//     finished beside the cells of layer k + 1;
//   * tiles of 16 x 16 cells, two CTAs of 256 threads per SM, so one computes while the other waits; the left
//     neighbour's contributions arrive by warp shuffle, the column's geometry stays in shared memory, so
//     that nothing spills (registers are the limit of the packed arithmetic: each value takes four).

// Measured (A apply, tile-line pass and interface included): level 7 / 129 layers 4.00 -> 2.17 ms, 6 / 65 0.51 ->
// 0.33 ms, with hourglass control 6 / 65 1.25 -> 0.46 ms; FMA pipes 55 % busy (43 % before, on 1.7 times the
// operations), the rest math-pipe throttle, dependent-issue waits and the barrier.  Error against binary64: 5.5e-15 in
// norm on random fields (3.5e-14 before), most of it from the 48-bit rounding of inputs and tables.

constexpr int kDfTI = 16, kDfTJ = 16, kDfThreads = kDfTI * kDfTJ;
constexpr int kDfNodes = (kDfTI + 1) * (kDfTJ + 1);
constexpr int kDfMaxKc = 64;  // cell layers per radial chunk at most
constexpr int kDfX = kDfTI + kDfTJ + 1;  // nodes of the tile's far row and column
constexpr int kDfCol = 2 * 3 * kDfTI;
// shared memory: per-node (s, d) of two layers (with hourglass control one, and one barrier more per layer); row
// sums (X, Y) of two layers; the column j0 + TJ's contributions of two layers; M^-1 and |det M| (and eL, eR) of
// the column; the chunk's layer constants; node values of two layers; the extra nodes' carry
constexpr size_t df_smem_bytes(bool hg) {
  return sizeof(float4) * (size_t)((hg ? 1 : 2) * 3 * kDfNodes + 2 * 3 * kDfThreads + 2 * kDfCol +
                                   (hg ? 12 : 10) * kDfThreads + 2 * (kDfMaxKc + 1)) +
         sizeof(double) * (size_t)(2 * 3 * kDfNodes + 3 * kDfX);
}
static_assert(df_smem_bytes(false) <= 113 * 1024 && df_smem_bytes(true) <= 113 * 1024, "two CTAs per SM");

__device__ __forceinline__ df2 df_from4(const float4& v) { return df2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 df_to4(const df2& a) { return make_float4(a.hi.x, a.hi.y, a.lo.x, a.lo.y); }

// One cell: sn = the (s, d) entry of corner 00, component 0; out(c, xy) takes (X, Y) of the corners 00, 10, 01,
// 11 of component c: bottom node X - Y, top node X + Y.  Arithmetic of OpA<T, HG>, lanes x = W0, y = W1.
// gc: the column's M^-1 (entries 0 .. 8), |det M| (9), eL, eR (10, 11); lc: (r, vol w0^2), (k9, vol w1^2).
template <bool HG, typename Out>
__device__ __forceinline__ void df_cell_A(const float4* sn, const float4* gc, const float4* lc, const dfl (&eta)[2],
                                          int div_term, const dfl& hgk, const Out& out) {
  const float4 l0 = lc[0], l1 = HG ? lc[1] : make_float4(0.f, 0.f, 0.f, 0.f);
  const df2 r = both(dfl(l0.x, l0.y)), vw2 = both(dfl(l0.z, l0.w));
  const df2 nk9 = both(dfl(-l1.x, -l1.y));
  df2 M[9], mr[3];
#pragma unroll
  for (int q = 0; q < 9; ++q) M[q] = df_from4(gc[q * kDfThreads]);
#pragma unroll
  for (int x = 0; x < 3; ++x) mr[x] = df_of(prod2(r, M[6 + x]));
  df2 G[3][3], b1[HG ? 3 : 1], b2[HG ? 3 : 1];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4* const s = sn + c * kDfNodes;
    const df2 n00 = df_from4(s[0]), n10 = df_from4(s[kDfTJ + 1]), n01 = df_from4(s[1]), n11 = df_from4(s[kDfTJ + 2]);
    const df2 n12 = df_of(sum2(n10, n01));  // (s, d) of 10 plus 01
    const df2 s0 = pack(lane_x(n00), lane_x(n11)), s1 = pack(lane_x(n10), lane_x(n01)),
              s2 = pack(lane_x(n01), lane_x(n10));
    // (normalised: after a cancellation their low part is large, and the products drop low x low)
    const df2 ax = norm2(diff2(s1, s0)), ay = norm2(diff2(s2, s0));
    const df2 d0 = pack(lane_y(n00), lane_y(n11));
    const df2 az = norm2(df_of(sum2(d0, both(lane_y(n12)))));
#pragma unroll
    for (int x = 0; x < 3; ++x) G[c][x] = dot3(ax, M[x], ay, M[3 + x], az, mr[x]);
    if constexpr (HG) {
      // b_1 = 2 alpha_1 - alpha_2 = (2 d_1 - d_2 - a_zeta / 3) - k9 (5 a_xi - 4 a_eta), b_2 with 1, 2 and
      // xi, eta exchanged
      const df2 d1 = pack(lane_y(n10), lane_y(n01)), d2 = pack(lane_y(n01), lane_y(n10));
      const df2 dd = diff2(d1, d2);
      acc2 a3 = prod2(az, both(dfl(-1.0 / 3.0)));
      acc2 p = a3, q = a3;
      acc_add2(p, dd), acc_add2(p, d1);
      acc_add2(q, neg2(dd)), acc_add2(q, d2);
      df2 dl = diff2(ax, ay);
      dl.hi = p2mul(dl.hi, make_float2(4.f, 4.f)), dl.lo = p2mul(dl.lo, make_float2(4.f, 4.f));
      acc_fma2(p, nk9, df_of(sum2(dl, ax)));
      acc_fma2(q, nk9, diff2(ay, dl));
      b1[c] = df_of(p), b2[c] = df_of(q);
    }
  }
  const df2 et = pack(eta[0], eta[1]);
  const df2 ve = mul2(mul2(vw2, df_from4(gc[9 * kDfThreads])), et);
  const df2 ve2{p2add(ve.hi, ve.hi), p2add(ve.lo, ve.lo)};  // exact doubling
  df2 S[3][3];
  if (div_term) {
    acc2 tr = sum2(G[0][0], G[1][1]);
    acc_add2(tr, G[2][2]);
    const acc2 vt = prod2(df_of(prod2(ve, both(dfl(-2.0 / 3.0)))), df_of(tr));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      acc2 a = vt;
      acc_fma2(a, ve2, G[c][c]);
      S[c][c] = norm2(df_of(a));
    }
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) S[c][c] = norm2(df_of(prod2(ve2, G[c][c])));
  }
  S[0][1] = S[1][0] = norm2(df_of(prod2(ve, df_of(sum2(G[0][1], G[1][0])))));
  S[0][2] = S[2][0] = norm2(df_of(prod2(ve, df_of(sum2(G[0][2], G[2][0])))));
  S[1][2] = S[2][1] = norm2(df_of(prod2(ve, df_of(sum2(G[1][2], G[2][1])))));
  df2 nek{}, e3{};
  if constexpr (HG) {
    acc2 g = prod2(vw2, df_from4(gc[10 * kDfThreads]));
    acc_fma2(g, both(dfl(l1.z, l1.w)), df_from4(gc[11 * kDfThreads]));
    const df2 eps = mul2(mul2(both(hgk), et), df_of(g));
    nek = df_of(prod2(eps, nk9)), e3 = df_of(prod2(eps, both(dfl(1.0 / 3.0))));
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    acc2 h0 = prod2(S[c][0], M[0]), h1 = prod2(S[c][0], M[3]);
    acc_fma2(h0, S[c][1], M[1]), acc_fma2(h1, S[c][1], M[4]);
    acc_fma2(h0, S[c][2], M[2]), acc_fma2(h1, S[c][2], M[5]);
    const df2 h2 = dot3(S[c][0], mr[0], S[c][1], mr[1], S[c][2], mr[2]);
    df2 y03 = h2, y12;
    if constexpr (HG) {
      acc_fma2(h0, nek, b1[c]), acc_fma2(h1, nek, b2[c]);
      acc2 y0 = acc_of(h2), y1 = y0, y2 = y0;
      const df2 ne3 = neg2(e3);
      acc_fma2(y0, ne3, df_of(sum2(b1[c], b2[c])));
      acc_fma2(y1, e3, b1[c]), acc_fma2(y2, e3, b2[c]);
      y03 = df_of(y0);
      // 10 = W0 node 1 + W1 node 2, 01 = W0 node 2 + W1 node 1
      const df2 f1 = df_of(y1), f2 = df_of(y2);
      y12 = df_of(sum2(pack(lane_x(f1), lane_x(f2)), pack(lane_y(f2), lane_y(f1))));
    } else {
      const df2 sw = pack(lane_y(h2), lane_x(h2));
      y12 = df_of(sum2(h2, sw));
    }
    const df2 H0 = df_of(h0), H1 = df_of(h1);
    const df2 x03 = neg2(df_of(sum2(H0, H1)));
    const df2 x12 = df_of(sum2(pack(lane_x(H0), lane_x(H1)), pack(lane_y(H1), lane_y(H0))));
    const df2 xy[4] = {pack(lane_x(x03), lane_x(y03)), pack(lane_x(x12), lane_x(y12)), pack(lane_y(x12), lane_y(y12)),
                       pack(lane_y(x03), lane_y(y03))};
    out(c, xy);
  }
}

__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

template <bool HG, int FLAGS, int EPI>
__global__ void __launch_bounds__(kDfThreads, 2)
    k_df_A(Dims D, int div_term, dfl hgk, const double* __restrict__ in0, const double* __restrict__ in1,
           const double* __restrict__ in2, double* __restrict__ out0, double* __restrict__ out1,
           double* __restrict__ out2, const double* __restrict__ geo, const dfl* __restrict__ lay,
           const double* __restrict__ eta, const double* __restrict__ svec, int bc_in, int bc_out, int kc,
           const int* __restrict__ skip, EpiArgs<double> E, double* __restrict__ ring) {
  constexpr int TI = kDfTI, TJ = kDfTJ, NT = kDfThreads;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  float4* const sd = reinterpret_cast<float4*>(tile_smem);  // [2 or 1][3][kDfNodes]
  float4* const sr = sd + (HG ? 1 : 2) * 3 * kDfNodes;      // [2][3][NT]
  float4* const scol = sr + 2 * 3 * NT;                     // [2][2][3][TI]
  float4* const gc = scol + 2 * kDfCol + threadIdx.x;       // [10 or 12][NT]
  float4* const lct = scol + 2 * kDfCol + (HG ? 12 : 10) * NT;               // [kDfMaxKc + 1][2]
  double* const raw = reinterpret_cast<double*>(lct + 2 * (kDfMaxKc + 1));   // [2][3][kDfNodes]
  float2* const xcarry = reinterpret_cast<float2*>(raw + 2 * 3 * kDfNodes);  // [3][kDfX]
  if (skip && *skip) return;
  const int N = D.N, n_r = D.n_r, P = D.P;
  const int LS = (int)D.layer_stride, NLL = (int)D.n_lat_layout;
  const RingDims RD = ring_dims(N, TI, TJ);
  const int ntj = N / TJ;
  const int i0 = (blockIdx.x / ntj) * TI, j0 = (blockIdx.x % ntj) * TJ;
  const int d = blockIdx.z;
  const int kc0 = blockIdx.y * kc, kc1 = min(n_r - 1, kc0 + kc);
  const int ti = threadIdx.x / TJ, tj = threadIdx.x % TJ;
  const int ci = i0 + ti, cj = j0 + tj;  // this thread's cell; its corner 00 is its own node
  const int dbase = (int)(d * D.diamond_stride), lbase = d * (N + 1) * P;
  const int c00 = dbase + ci * P + cj;
  {
    df2 M[9];
    const int t0 = ((d * N + ci) * N + cj) * 2, nt = (int)D.n_tri;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const double2 g = *reinterpret_cast<const double2*>(geo + q * nt + t0);  // t0 and nt are even
      M[q] = pack(split(g.x), split(g.y));
      gc[q * NT] = df_to4(M[q]);
    }
    const double2 g = *reinterpret_cast<const double2*>(geo + 9 * nt + t0);
    const df2 dM = pack(split(g.x), split(g.y));
    gc[9 * NT] = df_to4(dM);
    if constexpr (HG) {  // hg_column
      acc2 l = prod2(M[0], M[0]), qq = prod2(M[6], M[6]);
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const df2 s01 = df_of(sum2(M[x], M[3 + x]));
        if (x > 0) acc_fma2(l, M[x], M[x]), acc_fma2(qq, M[6 + x], M[6 + x]);
        acc_fma2(l, M[3 + x], M[3 + x]);
        acc_fma2(l, s01, s01);
      }
      gc[10 * NT] = df_to4(mul2(both(dfl(2.0)), mul2(dM, df_of(l))));
      gc[11 * NT] = df_to4(mul2(both(dfl(6.0)), mul2(dM, df_of(qq))));
    }
  }
  const double2* const etac = reinterpret_cast<const double2*>(eta) + ((int64_t)d * (n_r - 1) * N + ci) * N + cj;
  const int eta_ls = N * N;
  // the extra nodes of the tile (its far row and column): threads 0 .. NX - 1 keep one each beside their own
  constexpr int NX = kDfX;
  const bool hasx = (int)threadIdx.x < NX;
  const int xsi = (int)threadIdx.x <= TJ ? TI : (int)threadIdx.x - TJ - 1, xsj = (int)threadIdx.x <= TJ ? (int)threadIdx.x : TJ;
  const int x00 = dbase + (i0 + xsi) * P + j0 + xsj;

  const int slot0 = ti * (TJ + 1) + tj, slotx = xsi * (TJ + 1) + xsj;
  // request of this thread's node values of a layer (each thread reads back only what it copied)
  auto request = [&](int layer) {
    const uint32_t dst = smem_u32(raw + (layer & 1) * 3 * kDfNodes + slot0);
    const int o = c00 + layer * LS;
    cp_async8(dst, in0 + o), cp_async8(dst + 8 * kDfNodes, in1 + o), cp_async8(dst + 16 * kDfNodes, in2 + o);
    if (hasx) {
      const uint32_t dx = smem_u32(raw + (layer & 1) * 3 * kDfNodes + slotx);
      const int x = x00 + layer * LS;
      cp_async8(dx, in0 + x), cp_async8(dx + 8 * kDfNodes, in1 + x), cp_async8(dx + 16 * kDfNodes, in2 + x);
    }
    cp_async_commit();
  };
  // (s, d) = (top + bottom, top - bottom) of a node between layers k and k + 1, projected on the boundary layers
  auto put_node = [&](int k, int slot, int off) {
    double b[3], t[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      b[c] = raw[((k & 1) * 3 + c) * kDfNodes + slot];
      t[c] = raw[(((k + 1) & 1) * 3 + c) * kDfNodes + slot];
    }
    if (FLAGS & PROJ_IN) {
      const int64_t so = lbase + off - dbase;
      if (k == 0) project_vec(b, svec, so, (int64_t)NLL, bc_in);
      if (k + 1 == n_r - 1) project_vec(t, svec, so, (int64_t)NLL, bc_out);
    }
    float4* const s = sd + (HG ? 0 : k & 1) * 3 * kDfNodes + slot;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const dfl B = split(b[c]), T = split(t[c]);
      s[c * kDfNodes] = df_to4(df_of(sum2(both(T), pack(B, -B))));
    }
  };
  const int64_t ring_c = (int64_t)n_r * 10 * RD.RC;  // stride of one (slot, component)
  auto ring_store = [&](int k, int i, int j, int slot, const double (&v)[3]) {
    const int64_t base = (int64_t)k * 10 * RD.RC + (int64_t)d * RD.RC + ring_index(RD, N, i, j);
#pragma unroll
    for (int c = 0; c < 3; ++c) ring[(slot * 3 + c) * ring_c + base] = v[c];
  };
  auto store_node = [&](int k, double (&v)[3]) {  // this thread's own node, inside the tile
    const int idx = c00 + k * LS;
    if ((FLAGS & PROJ_OUT) && (k == 0 || k == n_r - 1)) {
      const int bc = k == 0 ? bc_in : bc_out;
      const int64_t so = lbase + ci * P + cj;
      project_vec(v, svec, so, (int64_t)NLL, bc);
      if (FLAGS & ADD_ID) {
        double uu[3] = {in0[idx], in1[idx], in2[idx]};
        double pu[3] = {uu[0], uu[1], uu[2]};
        project_vec(pu, svec, so, (int64_t)NLL, bc);
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] += uu[c] - pu[c];
      }
    }
    if (EPI != EPI_NONE) {
      epilogue<double, EPI>(E, in0, in1, in2, idx, v);
      return;
    }
    out0[idx] = v[0], out1[idx] = v[1], out2[idx] = v[2];
  };
  const bool interior = ti >= 1 && tj >= 1;
  auto emit = [&](int k, const df2 (&v)[2]) {  // own node: components (0, 1), (2, -)
    double o[3] = {join(lane_x(v[0])), join(lane_y(v[0])), join(lane_x(v[1]))};
    if (interior) store_node(k, o);
    else ring_store(k, ci, cj, 2 * (ti == 0) + (tj == 0), o);
  };
  auto emit_x = [&](int k, const df2 (&v)[2]) {
    const double o[3] = {join(lane_x(v[0])), join(lane_y(v[0])), join(lane_x(v[1]))};
    ring_store(k, i0 + xsi, j0 + xsj, 2 * (xsi == 0) + (xsj == 0), o);
  };
  // lateral sums (X, Y) of a node -> its value v = X - Y + carry (bottom) and the new carry X + Y
  auto radial = [&](const acc2 (&a)[3], df2 (&carry)[2], df2 (&v)[2]) {
    df2 bt[3];  // (X - Y, X + Y)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const df2 xyv = df_of(a[c]);
      const dfl X = lane_x(xyv), Y = lane_y(xyv);
      bt[c] = df_of(sum2(both(X), pack(-Y, Y)));
    }
    v[0] = df_of(sum2(pack(lane_x(bt[0]), lane_x(bt[1])), carry[0]));
    v[1] = df_of(sum2(both(lane_x(bt[2])), carry[1]));
    carry[0] = pack(lane_y(bt[0]), lane_y(bt[1]));
    carry[1] = both(lane_y(bt[2]));
  };
  auto get_xcarry = [&](df2 (&xc)[2]) {
    const float2 p = xcarry[threadIdx.x], q = xcarry[NX + threadIdx.x], r = xcarry[2 * NX + threadIdx.x];
    xc[0] = pack(dfl(p.x, p.y), dfl(q.x, q.y)), xc[1] = both(dfl(r.x, r.y));
  };
  // a value of the left neighbour (i, j - 1), zero at the tile's first column
  auto left = [&](const df2& a) {
    df2 r{make_float2(__shfl_up_sync(0xffffffffu, a.hi.x, 1, TJ), __shfl_up_sync(0xffffffffu, a.hi.y, 1, TJ)),
          make_float2(__shfl_up_sync(0xffffffffu, a.lo.x, 1, TJ), __shfl_up_sync(0xffffffffu, a.lo.y, 1, TJ))};
    if (tj == 0) r = both(dfl(0.f, 0.f));
    return r;
  };

  const int kstart = kc0 > 0 ? kc0 - 1 : 0;
  const df2 zero = both(dfl(0.f, 0.f));
  df2 carry[2] = {zero, zero};
  if (hasx)
#pragma unroll
    for (int c = 0; c < 3; ++c) xcarry[c * NX + threadIdx.x] = make_float2(0.f, 0.f);
  request(kstart), request(kstart + 1);
  cp_async_wait<0>();
  put_node(kstart, slot0, c00);
  if (hasx) put_node(kstart, slotx, x00);
  double2 en = etac[(int64_t)kstart * eta_ls];
  for (int t = threadIdx.x; t < kc1 - kstart; t += NT) {
    const dfl* l = lay + kLayerStride * (kstart + t);
    lct[2 * t] = make_float4(l[4].hi, l[4].lo, l[5].hi, l[5].lo);
    lct[2 * t + 1] = make_float4(l[8].hi, l[8].lo, l[9].hi, l[9].lo);
  }
  __syncthreads();
  for (int k = kstart; k < kc1; ++k) {
    // requests of the next layer, in flight during the cell arithmetic
    const double2 ek = en;
    const bool more = k + 1 < kc1;
    if (more) {
      request(k + 2);
      en = etac[(int64_t)(k + 1) * eta_ls];
    }
    if (TN_EPI_PREFETCH && EPI != EPI_NONE && interior && k >= kc0) {
      const int idx = c00 + k * LS;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (EPI == EPI_CHEB2) prefetch_l1(E.r[c] + idx), prefetch_l1(E.xacc[c] + idx);
        else prefetch_l1(E.b[c] + idx);
      }
      if (EPI != EPI_RESID)
#pragma unroll
        for (int q = 0; q < 6; ++q) prefetch_l1(E.binv[q] + idx);
    }
    // row sums: own corner 00 with the left cell's 01 (kept), own 10 with the left cell's 11 (for the row below)
    float4* const rs = sr + (k & 1) * 3 * NT;
    float4* const cs = scol + (k & 1) * kDfCol;
    acc2 a[3];
    {
      const dfl e[2] = {split(ek.x), split(ek.y)};
      df_cell_A<HG>(sd + (HG ? 0 : k & 1) * 3 * kDfNodes + slot0, gc, lct + 2 * (k - kstart), e, div_term, hgk,
                    [&](int c, const df2 (&xy)[4]) {
                      if (tj == TJ - 1) cs[c * TI + ti] = df_to4(xy[2]), cs[(3 + c) * TI + ti] = df_to4(xy[3]);
                      a[c] = sum2(xy[0], left(xy[2]));
                      rs[c * NT + threadIdx.x] = df_to4(df_of(sum2(xy[1], left(xy[3]))));
                    });
    }
    if (HG) __syncthreads();  // every thread has read this layer's (s, d)
    if (more) {
      cp_async_wait<0>();
      put_node(k + 1, slot0, c00);
      if (hasx) put_node(k + 1, slotx, x00);
    }
    // the arrays that layer k + 1 writes were last read before the previous barrier (layer k - 1's cells and
    // nodes), so one barrier per layer separates every write from its readers
    __syncthreads();
    df2 v[2];
    if (ti >= 1) {
#pragma unroll
      for (int c = 0; c < 3; ++c) acc_add2(a[c], df_from4(rs[c * NT + threadIdx.x - TJ]));
    }
    radial(a, carry, v);
    if (k >= kc0) emit(k, v);
    if (hasx) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (xsj < TJ) {  // far row: the last row's sums
          a[c] = acc_of(df_from4(rs[c * NT + (TI - 1) * TJ + xsj]));
        } else {  // far column: corner 01 of the row, corner 11 of the row above
          a[c] = acc_of(xsi < TI ? df_from4(cs[c * TI + xsi]) : zero);
          if (xsi >= 1) acc_add2(a[c], df_from4(cs[(3 + c) * TI + xsi - 1]));
        }
      }
      df2 xc[2];
      get_xcarry(xc);
      radial(a, xc, v);
      const float2 n[3] = {make_float2(xc[0].hi.x, xc[0].lo.x), make_float2(xc[0].hi.y, xc[0].lo.y),
                           make_float2(xc[1].hi.x, xc[1].lo.x)};
#pragma unroll
      for (int c = 0; c < 3; ++c) xcarry[c * NX + threadIdx.x] = n[c];
      if (k >= kc0) emit_x(k, v);
    }
  }
  if (kc1 == n_r - 1) {
    emit(n_r - 1, carry);
    if (hasx) {
      df2 xc[2];
      get_xcarry(xc);
      emit_x(n_r - 1, xc);
    }
  }
}
