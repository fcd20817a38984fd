// Double-float diag(A) of FP64 levels with N >= 32 (included by kernels.cu inside its namespace, after k_diag_A).
//
// OpDiag's factor table, without or with hourglass control.  Summed over the two cell layers
// around node layer k first, triangle t gives its local node a the diagonal entries
//   P_ad alpha + Q_d beta + 2 R_ad gamma,   alpha = A_k + A_k-1,  beta = r_k^2 A_k + r_k-1^2 A_k-1,
//   gamma = r_k-1 A_k-1 - r_k A_k,   A_k = vol w0^2 |det M| eta,
// so a cell does 21 products per node layer instead of 39 per cell layer and no contributions are carried.  The 21
// factors of the cell's two triangles stay in shared memory (k_tile_hf read them from L2 on every layer).
// The two boundary layers' nodes (k_diag_A's gather, FP64 pipe) run as CTAs of the same launch (blockIdx.y 0 and 1)
// beside the FP32 work of the others.
// Measured, level 7 / 129 layers: element kernel and boundary gather 1.62 + 0.16 ms -> 0.77 ms; FP32 pipe and its
// dependent-issue waits.  Error against 64 bits 2.4e-14 -> 3e-15.
constexpr int kDgRow = 2, kDgMaxKc = 64;
constexpr size_t df_diag_smem(bool hg) {
  return sizeof(float4) * (size_t)((hg ? 23 : 21) * kDfThreads + 2 * kDgRow * kDfThreads + 2 * 2 * kDgRow * kDfTI +
                                   2 * (kDgMaxKc + 1));
}
static_assert(df_diag_smem(true) <= 113 * 1024, "two CTAs per SM");

template <bool HG>
__global__ void __launch_bounds__(kDfThreads, 2)
    k_df_diag(Dims D, dfl hgk, DiagBoundary<double> B, double* __restrict__ d0, double* __restrict__ d1,
              double* __restrict__ d2, const float4* __restrict__ coef, int n_pair, const dfl* __restrict__ lay,
              const double* __restrict__ eta, int kc, double* __restrict__ ring) {
  constexpr int TI = kDfTI, TJ = kDfTJ, NT = kDfThreads, NX = kDfX;
  const int N = D.N, n_r = D.n_r, P = D.P, d = blockIdx.z;
  if (blockIdx.y < 2) {
    for (int t = (int)(blockIdx.x * NT + threadIdx.x); t < (N + 1) * (N + 1); t += (int)gridDim.x * NT)
      diag_boundary_node<double>(D, B, t, (int)blockIdx.y, d, d0, d1, d2);
    return;
  }
  extern __shared__ __align__(16) unsigned char tile_smem[];
  df2* const cf = reinterpret_cast<df2*>(tile_smem) + threadIdx.x;                        // [21 or 23][NT]
  df2* const sr = reinterpret_cast<df2*>(tile_smem) + (HG ? 23 : 21) * NT;                // [2][2][NT]
  df2* const scol = sr + 2 * kDgRow * NT;                                                 // [2][2][2][TI]
  float4* const lct = reinterpret_cast<float4*>(scol + 2 * 2 * kDgRow * TI);             // [kDgMaxKc + 1][2]
  const RingDims RD = ring_dims(N, TI, TJ);
  const int ntj = N / TJ;
  const int i0 = (blockIdx.x / ntj) * TI, j0 = (blockIdx.x % ntj) * TJ;
  const int ti = threadIdx.x / TJ, tj = threadIdx.x % TJ, ci = i0 + ti, cj = j0 + tj;
  // node layers kn0 .. kn1 - 1 of 1 .. n_r - 2
  const int kn0 = 1 + ((int)blockIdx.y - 2) * kc, kn1 = min(n_r - 1, kn0 + kc);
  const int p0 = (d * N + ci) * N + cj;
#pragma unroll
  for (int q = 0; q < (HG ? 23 : 21); ++q) cf[q * NT] = df_from4(coef[(int64_t)q * n_pair + p0]);
  for (int t = threadIdx.x; t <= kn1 - kn0; t += NT) {  // cell layers kn0 - 1 .. kn1 - 1
    const dfl* l = lay + kLayerStride * (kn0 - 1 + t);
    lct[2 * t] = make_float4(l[4].hi, l[4].lo, l[5].hi, l[5].lo);
    lct[2 * t + 1] = make_float4(l[8].hi, l[8].lo, l[9].hi, l[9].lo);
  }
  df2 dM;
  {
    const double2 g = *reinterpret_cast<const double2*>(B.geo + 9 * D.n_tri + 2 * (int64_t)p0);
    dM = pack(split(g.x), split(g.y));
  }
  const double2* const etac = reinterpret_cast<const double2*>(eta) + ((int64_t)d * (n_r - 1) * N + ci) * N + cj;
  const int eta_ls = N * N;
  const bool hasx = (int)threadIdx.x < NX;
  const int xsi = (int)threadIdx.x <= TJ ? TI : (int)threadIdx.x - TJ - 1, xsj = (int)threadIdx.x <= TJ ? (int)threadIdx.x : TJ;
  const bool interior = ti >= 1 && tj >= 1;
  const int64_t ring_c = (int64_t)n_r * 10 * RD.RC;
  auto ring_store = [&](int k, int i, int j, int slot, const double (&v)[3]) {
    const int64_t base = (int64_t)k * 10 * RD.RC + (int64_t)d * RD.RC + ring_index(RD, N, i, j);
#pragma unroll
    for (int c = 0; c < 3; ++c) ring[(slot * 3 + c) * ring_c + base] = v[c];
  };
  // A, r A, r^2 A of a cell layer (and eps (k9 +/- 1/3)^2 with hourglass control: as the bottom, as the top layer)
  struct Cell {
    df2 A, B, C, eb, et;
  };
  auto cell = [&](int k, const double2& e, Cell& s) {
    const float4 l0 = lct[2 * (k - kn0 + 1)];
    const df2 r = both(dfl(l0.x, l0.y)), vw2 = both(dfl(l0.z, l0.w));
    const df2 et = df_of(prod2(dM, pack(split(e.x), split(e.y))));
    s.A = mul2(vw2, et), s.B = df_of(prod2(r, s.A)), s.C = df_of(prod2(r, s.B));
    if constexpr (HG) {
      const float4 l1 = lct[2 * (k - kn0 + 1) + 1];
      const df2 k9 = both(dfl(l1.x, l1.y)), third = both(dfl(1.0 / 3.0));
      acc2 g = prod2(vw2, cf[21 * NT]);
      acc_fma2(g, both(dfl(l1.z, l1.w)), cf[22 * NT]);
      const df2 eps = mul2(mul2(both(hgk), et), df_of(g));
      const df2 kb = df_of(sum2(k9, third)), kt = diff2(k9, third);
      s.eb = df_of(prod2(eps, mul2(kb, kb))), s.et = df_of(prod2(eps, mul2(kt, kt)));
    }
  };
  auto left = [&](const df2& a) {  // the left neighbour's value, zero at the tile's first column
    df2 r{make_float2(__shfl_up_sync(0xffffffffu, a.hi.x, 1, TJ), __shfl_up_sync(0xffffffffu, a.hi.y, 1, TJ)),
          make_float2(__shfl_up_sync(0xffffffffu, a.lo.x, 1, TJ), __shfl_up_sync(0xffffffffu, a.lo.y, 1, TJ))};
    if (tj == 0) r = both(dfl(0.f, 0.f));
    return r;
  };
  __syncthreads();
  Cell prev;
  cell(kn0 - 1, etac[(int64_t)(kn0 - 1) * eta_ls], prev);
  double2 en = etac[(int64_t)kn0 * eta_ls];
  for (int k = kn0; k < kn1; ++k) {
    const double2 ek = en;
    if (k + 1 < kn1) en = etac[(int64_t)(k + 1) * eta_ls];
    Cell cur;
    cell(k, ek, cur);
    const df2 al = df_of(sum2(cur.A, prev.A)), be = df_of(sum2(cur.C, prev.C));
    df2 ga = diff2(prev.B, cur.B);
    ga.hi = p2add(ga.hi, ga.hi), ga.lo = p2add(ga.lo, ga.lo);
    df2 n2{}, n5{};  // hourglass part of local nodes 0 and 1, 2
    if constexpr (HG) {
      const df2 s = df_of(sum2(cur.eb, prev.et));
      n2 = df2{p2add(s.hi, s.hi), p2add(s.lo, s.lo)};
      n5 = df_of(sum2(df2{p2add(n2.hi, n2.hi), p2add(n2.lo, n2.lo)}, s));
      prev.et = cur.et;
    }
    prev.A = cur.A, prev.B = cur.B, prev.C = cur.C;
    dfl own[3], row[3], c01[3], c11[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const acc2 qb = prod2(cf[(18 + c) * NT], be);
      df2 v[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        acc2 s = qb;
        if constexpr (HG) acc_add2(s, a == 0 ? n2 : n5);
        acc_fma2(s, cf[(3 * a + c) * NT], al);
        acc_fma2(s, cf[(9 + 3 * a + c) * NT], ga);
        v[a] = df_of(s);
      }
      // corners 00 = W0 node 0, 11 = W1 node 0, 10 = W0 node 1 + W1 node 2, 01 = W0 node 2 + W1 node 1
      const df2 m = df_of(sum2(pack(lane_x(v[1]), lane_x(v[2])), pack(lane_y(v[2]), lane_y(v[1]))));
      c01[c] = lane_y(m), c11[c] = lane_y(v[0]);
      // (00, 10) plus the left cell's (01, 11)
      const df2 s = df_of(sum2(pack(lane_x(v[0]), lane_x(m)), left(pack(c01[c], c11[c]))));
      own[c] = lane_x(s), row[c] = lane_y(s);
    }
    df2* const rs = sr + (k & 1) * kDgRow * NT;
    df2* const cs = scol + (k & 1) * 2 * kDgRow * TI;
    rs[threadIdx.x] = pack(row[0], row[1]), rs[NT + threadIdx.x] = both(row[2]);
    if (tj == TJ - 1) {
      cs[ti] = pack(c01[0], c01[1]), cs[TI + ti] = both(c01[2]);
      cs[2 * TI + ti] = pack(c11[0], c11[1]), cs[3 * TI + ti] = both(c11[2]);
    }
    __syncthreads();  // the arrays of layer k + 1 were last read before it
    {
      df2 a = pack(own[0], own[1]), b = both(own[2]);
      if (ti >= 1) a = df_of(sum2(a, rs[threadIdx.x - TJ])), b = df_of(sum2(b, rs[NT + threadIdx.x - TJ]));
      const double o[3] = {join(lane_x(a)), join(lane_y(a)), join(lane_x(b))};
      if (interior) {
        const int idx = (int)(d * D.diamond_stride) + k * (int)D.layer_stride + ci * P + cj;
        d0[idx] = o[0], d1[idx] = o[1], d2[idx] = o[2];
      } else {
        ring_store(k, ci, cj, 2 * (ti == 0) + (tj == 0), o);
      }
    }
    if (hasx) {
      const df2 zero = both(dfl(0.f, 0.f));
      df2 a, b;
      if (xsj < TJ) {  // far row: the last row's sums
        a = rs[(TI - 1) * TJ + xsj], b = rs[NT + (TI - 1) * TJ + xsj];
      } else {  // far column: corner 01 of the row, corner 11 of the row above
        a = xsi < TI ? cs[xsi] : zero, b = xsi < TI ? cs[TI + xsi] : zero;
        if (xsi >= 1) a = df_of(sum2(a, cs[2 * TI + xsi - 1])), b = df_of(sum2(b, cs[3 * TI + xsi - 1]));
      }
      const double o[3] = {join(lane_x(a)), join(lane_y(a)), join(lane_x(b))};
      ring_store(k, i0 + xsi, j0 + xsj, 2 * (xsi == 0) + (xsj == 0), o);
    }
  }
}
