// Heun steps with a fixed velocity as a stencil (included by energy.cu inside its namespace).
//
// The residual R = (K + C(u) + S(u)) T is linear in T, and u is fixed over the steps of one call: so the rows of the
// matrix are assembled once per call and every residual is a 21-point stencil (7 lateral x 3 radial nodes).  The
// element-by-element residual spends about 440 FP64 instructions per cell (cbrt, tanh, divisions for tau; 1.9 ms at
// level 6 / 65 layers, the FP64 pipe); a stencil residual reads 160 bytes per node and does 40 FP64
// instructions.  Constants are in the null space of all three terms, so the rows hold no diagonal and act on
// differences to the node's own value: exactly zero for constants, and no cancellation of large T.
// Measured, level 6 / 65 layers: ten Heun steps 39.9 -> 7.1 ms (wedge values 0.73 ms, rows 1.7 ms, 0.23 ms per stage,
// all held by the FP64 pipe); one step 4.0 -> 2.9 ms.
// Nodes that several diamonds share keep one partial row per copy (the wedges of that diamond).

struct RowDims {
  int N, n_r, P, ls, n_groups, n_lat;
  int64_t ds, n;  // diamond stride, layout entries
  const int* gptr;
  const int64_t* goff;
};
inline RowDims row_dims(const Level& L) {
  return RowDims{L.N, L.n_r, L.P, (int)L.layer_stride, L.n_groups, 10 * L.N * L.N + 2, L.diamond_stride, L.n_layout,
                 L.grp_ptr, L.grp_off};
}

constexpr int kRowCoef = 20;  // radial -1: lateral 0 .. 6; radial 0: 1 .. 6; radial +1: 0 .. 6
// lateral neighbours 0 .. 6: the node, (1,0) (0,1) (-1,1) (-1,0) (0,-1) (1,-1)
__device__ constexpr int kNbI[7] = {0, 1, 0, -1, -1, 0, 1}, kNbJ[7] = {0, 0, 1, 1, 0, -1, -1};
// the six triangles around a node: cell offset, wedge, lateral neighbour of its local nodes 0, 1, 2
__device__ constexpr int kRowTri[6][6] = {{0, 0, 0, 0, 1, 2},   {-1, 0, 1, 2, 3, 0}, {-1, 0, 0, 4, 0, 3},
                                          {-1, -1, 1, 0, 4, 5}, {0, -1, 0, 5, 6, 0}, {0, -1, 1, 1, 0, 6}};

// psi(z) = (x coth x - 1) / x^2, z = x^2: tau = h^2 / 4 psi(Pe^2).  Lambert's continued fraction of tanh,
// psi = 1 / (3 + z / (5 + z / (7 + ... ))), cut after 14 terms, as a quotient of polynomials up to z = 16 (truncation
// 1e-17, all coefficients positive), the definition beyond (no cancellation there).
__device__ __forceinline__ double supg_psi(double z) {
  if (z > 16.0) {
    const double x = sqrt(z), e = exp(-2.0 * x);
    return (x * ((1.0 + e) / (1.0 - e)) - 1.0) / z;
  }
  double p = 119.0, q = 1.0;
  p = p * z + 271320.0, q = q * z + 7140.0;
  p = p * z + 166658310.0, q = q * z + 7936110.0;
  p = p * z + 40156716600.0, q = q * z + 3055402350.0;
  p = p * z + 4141161399375.0, q = q * z + 496939367925.0;
  p = p * z + 170766437341500.0, q = q * z + 34785755754750.0;
  p = p * z + 2063427784543125.0, q = q * z + 924984868933125.0;
  q = q * z + 6190283353629375.0;
  return p / q;
}

// Per wedge (wedge layout): V tau, w0 ubar . m0, w0 ubar . m1, w0 r ubar . m2 (rows of M^-1).  One thread per lateral
// wedge and a few cell layers.
constexpr int kWedgeLayers = 4;
__global__ void __launch_bounds__(128) k_energy_wedge(Dims D, const double* __restrict__ geo, const double* __restrict__ lay,
                                                      const double* __restrict__ u0, const double* __restrict__ u1,
                                                      const double* __restrict__ u2, int supg, WedgeFlow* __restrict__ wq) {
  const int N = D.N, t = blockIdx.x * 128 + threadIdx.x;  // grid: lateral wedges x layer groups x 10 diamonds
  if (t >= 2 * N * N) return;
  const int i = t / (2 * N), r0 = t - i * 2 * N, j = r0 >> 1, w = r0 & 1, d = blockIdx.z;
  const int k0 = blockIdx.y * kWedgeLayers, k1 = min(D.n_r - 1, k0 + kWedgeLayers);
  const int64_t lt = (int64_t)d * 2 * N * N + t;
  double M[9];
  for (int q = 0; q < 9; ++q) M[q] = geo[(int64_t)q * D.n_tri + lt];
  const double dM = geo[9 * D.n_tri + lt], cd = cbrt(2.0 * dM);
  const int a[3][2] = {{w ? i + 1 : i, w ? j + 1 : j}, {w ? i : i + 1, w ? j + 1 : j}, {w ? i + 1 : i, w ? j : j + 1}};
  const double* u[3] = {u0, u1, u2};
  auto sum3 = [&](int k, double (&s)[3]) {
    const int64_t b = (int64_t)d * D.diamond_stride + (int64_t)k * D.layer_stride;
    for (int c = 0; c < 3; ++c)
      s[c] = (u[c][b + a[0][0] * D.P + a[0][1]] + u[c][b + a[1][0] * D.P + a[1][1]]) + u[c][b + a[2][0] * D.P + a[2][1]];
  };
  double lo[3], hi[3];
  sum3(k0, lo);
  for (int k = k0; k < k1; ++k) {
    sum3(k + 1, hi);
    double ub[3], un2 = 0;
    for (int c = 0; c < 3; ++c) ub[c] = (lo[c] + hi[c]) * (1.0 / 6.0), un2 += ub[c] * ub[c], lo[c] = hi[c];
    const double* l = lay + kLayerStride * k;
    const double w0 = l[0], vol = l[2], r = l[4];
    double vt = 0;
    if (supg) {
      const double h = cbrt(vol) * cd, h2 = 0.25 * (h * h);  // h = (2 V)^(1/3)
      vt = vol * dM * (h2 * supg_psi(un2 * h2));
    }
    const double m0 = (ub[0] * M[0] + ub[1] * M[1]) + ub[2] * M[2], m1 = (ub[0] * M[3] + ub[1] * M[4]) + ub[2] * M[5],
                 m2 = (ub[0] * M[6] + ub[1] * M[7]) + ub[2] * M[8];
    wq[((int64_t)d * (D.n_r - 1) + k) * 2 * N * N + t] = WedgeFlow{vt, w0 * m0, w0 * m1, (w0 * r) * m2};
  }
}

// Rows dt / m_j (K + C + S)_j of the interior node layers, thread per layout node.  Node j = (local a, side s) of
// wedge (t, k) has, with A = V w0^2, beta_a,s = lam_a + s mu (w0 ubar . grad) and C = V / 6 + V tau beta_a,s, the entries
//   (b, s'):  P_b + s' Q,  P_b = A (l_a . l_b + s r l_b . m2) + C lam_b,  Q = A (r l_a . m2 + s r^2 |m2|^2) + C mu.
// The sums over the wedges run over P_b and Q apart, per side (three and five fused operations per wedge, side and b; adding
// P - Q and P + Q to the 21 entries took seven), and the dot products of a column's M^-1 rows serve kRowLayers node layers:
// about 350 FP64 instructions a node instead of 770.  2.3 -> 1.7 ms at level 6 / 65 layers; ten Heun steps 7.73 -> 7.11 ms, at
// level 4 / 17 layers 767 -> 760 us.
constexpr int kRowLayers = 8;  // at most: fewer where the grid would not give every SM three CTAs
__global__ void __launch_bounds__(128, 3) k_energy_rows(Dims D, int nk, const double* __restrict__ geo, const double* __restrict__ lay,
                                                     const WedgeFlow* __restrict__ wq, const double* __restrict__ mass,
                                                     double dt, int64_t n, double* __restrict__ rows) {
  const int N = D.N, M1 = N + 1;
  const int p = blockIdx.x * 128 + threadIdx.x;  // grid: lattice points x groups of interior node layers x 10 diamonds
  if (p >= M1 * M1) return;
  const int i = p / M1, j = p - i * M1, d = blockIdx.z;
  const int k0 = 1 + blockIdx.y * nk, k1 = min(D.n_r - 1, k0 + nk);
  bool on[6];
  double lr[6][2], nr[6][2], gg[6], dM[6];  // l_a . l_1, l_a . l_2 (l_0 = -(l_1 + l_2)), the same with m2, |m2|^2, |det M|
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int ci = i + kRowTri[q][0], cj = j + kRowTri[q][1];
    on[q] = ci >= 0 && cj >= 0 && ci < N && cj < N;
    lr[q][0] = lr[q][1] = nr[q][0] = nr[q][1] = gg[q] = dM[q] = 0.0;
    if (!on[q]) continue;
    const int a = kRowTri[q][3] == 0 ? 0 : (kRowTri[q][4] == 0 ? 1 : 2);
    const int64_t lt = (int64_t)d * 2 * N * N + (ci * N + cj) * 2 + kRowTri[q][2];
    double m[9];
#pragma unroll
    for (int x = 0; x < 9; ++x) m[x] = geo[(int64_t)x * D.n_tri + lt];
    dM[q] = geo[9 * D.n_tri + lt];
    const double g00 = m[0] * m[0] + m[1] * m[1] + m[2] * m[2], g01 = m[0] * m[3] + m[1] * m[4] + m[2] * m[5],
                 g11 = m[3] * m[3] + m[4] * m[4] + m[5] * m[5];
    nr[q][0] = m[0] * m[6] + m[1] * m[7] + m[2] * m[8], nr[q][1] = m[3] * m[6] + m[4] * m[7] + m[5] * m[8];
    gg[q] = m[6] * m[6] + m[7] * m[7] + m[8] * m[8];
    lr[q][0] = a == 0 ? -(g00 + g01) : (a == 1 ? g00 : g01), lr[q][1] = a == 0 ? -(g01 + g11) : (a == 1 ? g01 : g11);
  }
  for (int k = k0; k < k1; ++k) {
    double P[2][7], Q[2][7];  // [side][lateral neighbour], side 0: the node is on the wedge's bottom layer
#pragma unroll
    for (int x = 0; x < 7; ++x) P[0][x] = P[1][x] = Q[0][x] = Q[1][x] = 0.0;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      if (!on[q]) continue;
      const int a = kRowTri[q][3] == 0 ? 0 : (kRowTri[q][4] == 0 ? 1 : 2);
      const int t = ((i + kRowTri[q][0]) * N + j + kRowTri[q][1]) * 2 + kRowTri[q][2];
      const double ll[3] = {-(lr[q][0] + lr[q][1]), lr[q][0], lr[q][1]}, nm[3] = {-(nr[q][0] + nr[q][1]), nr[q][0], nr[q][1]};
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int kk = k - side;
        const double* l = lay + kLayerStride * kk;
        const WedgeFlow v = wq[((int64_t)d * (D.n_r - 1) + kk) * 2 * N * N + t];
        const double lam[3] = {-(v.l0 + v.l1), v.l0, v.l1}, r = l[4], A = l[5] * dM[q], V = l[2] * dM[q];
        const double sr = side ? r : -r, beta = lam[a] + (side ? v.mu : -v.mu), C = V * (1.0 / 6.0) + v.vt * beta;
        const double q0 = (A * r) * (nm[a] + sr * gg[q]) + C * v.mu;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const int nb = kRowTri[q][3 + b];
          P[side][nb] += A * (ll[b] + sr * nm[b]);
          P[side][nb] += C * lam[b];
          Q[side][nb] += q0;
        }
      }
    }
    const int64_t idx = (int64_t)d * D.diamond_stride + (int64_t)k * D.layer_stride + (int64_t)i * D.P + j;
    const double f = dt / mass[idx];
#pragma unroll
    for (int x = 0; x < 7; ++x) {
      rows[(int64_t)x * n + idx] = f * (P[1][x] - Q[1][x]);
      if (x > 0) rows[(int64_t)(6 + x) * n + idx] = f * ((P[1][x] + Q[1][x]) + (P[0][x] - Q[0][x]));
      rows[(int64_t)(13 + x) * n + idx] = f * (P[0][x] + Q[0][x]);
    }
  }
}

// One Heun stage over the unique lateral points: with d = dt M^-1 R(X), stage 1: out = X - d; stage 2: out = ((T + X) -
// d) / 2 (X = T*); surface layers keep X (stage 1) or are left alone (stage 2 writes T in place).
template <int STAGE>
__global__ void __launch_bounds__(256) k_energy_stage(RowDims S, const double* __restrict__ X, const double* T,
                                                      const double* __restrict__ rows, double* out) {
  const int g = blockIdx.x * 256 + threadIdx.x, k = blockIdx.y;  // grid: unique lateral points x n_r
  if (g >= S.n_lat) return;
  const bool surface = k == 0 || k == S.n_r - 1;
  if (surface && STAGE == 2) return;
  const int N = S.N, n1 = N - 1, in = 10 * n1 * n1;
  // points inside the diamonds first (whole rows of threads without copies), then the interface groups
  if (g < in) {
    const int d = g / (n1 * n1), r = g - d * n1 * n1, i = r / n1 + 1, j = r - (i - 1) * n1 + 1;
    const int64_t o = (int64_t)d * S.ds + (int64_t)k * S.ls + (int64_t)i * S.P + j;
    const double x = X[o];
    if (surface) {
      out[o] = x;
      return;
    }
    double s = 0.0;
#pragma unroll
    for (int q = 0; q <= kRowCoef; ++q) {
      if (q == 7) continue;
      const double y = X[o + (q / 7 - 1) * (int64_t)S.ls + kNbI[q % 7] * S.P + kNbJ[q % 7]];
      s += rows[(int64_t)(q < 7 ? q : q - 1) * S.n + o] * (y - x);
    }
    out[o] = STAGE == 1 ? x - s : 0.5 * ((T[o] + x) - s);
    return;
  }
  const int b = S.gptr[g - in], e = S.gptr[g - in + 1];
  const int64_t lo = (int64_t)k * S.ls;
  const double x = X[S.goff[b] + lo];
  double s = 0.0;
  if (!surface) {
    for (int c = b; c < e; ++c) {  // copies in ascending layout order
      const int64_t o = S.goff[c] + lo;
      const int r = (int)(S.goff[c] % S.ds), i = r / S.P, j = r - i * S.P;
      for (int q = 0; q <= kRowCoef; ++q) {
        if (q == 7) continue;
        const int ni = i + kNbI[q % 7], nj = j + kNbJ[q % 7];
        if (ni < 0 || nj < 0 || ni > N || nj > N) continue;
        const double y = X[o + (q / 7 - 1) * (int64_t)S.ls + (ni - i) * S.P + (nj - j)];
        s += rows[(int64_t)(q < 7 ? q : q - 1) * S.n + o] * (y - x);
      }
    }
  }
  const double v = surface ? x : (STAGE == 1 ? x - s : 0.5 * ((T[S.goff[b] + lo] + x) - s));
  for (int c = b; c < e; ++c) out[S.goff[c] + lo] = v;
}

// n Heun steps of T (in place) through the rows; T1: scratch of the node layout.
inline cudaError_t heun_rows(EnergyState& S, const Level& L, double* T, double* T1, const double* const* u, double dt,
                             int n, int supg, cudaStream_t st) {
  const Dims D = dims(L);
  const unsigned nt = (unsigned)((2 * L.N * L.N + 127) / 128), np = (unsigned)(((L.N + 1) * (L.N + 1) + 127) / 128);
  k_energy_wedge<<<dim3(nt, (L.n_r - 1 + kWedgeLayers - 1) / kWedgeLayers, 10), 128, 0, st>>>(
      D, L.geo64, L.lay64, u[0], u[1], u[2], supg, S.ws.wq);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    const int nk = std::max(1, std::min(kRowLayers, (int)(np * 10 * (L.n_r - 2) / (152 * 3))));
    k_energy_rows<<<dim3(np, (L.n_r - 2 + nk - 1) / nk, 10), 128, 0, st>>>(D, nk, L.geo64, L.lay64, S.ws.wq, S.mass, dt, L.n_layout,
                                                                          S.ws.rows);
    e = cudaGetLastError();
  }
  const RowDims R = row_dims(L);
  const dim3 grid((unsigned)((R.n_lat + 255) / 256), L.n_r);
  for (int s = 0; s < n && e == cudaSuccess; ++s) {
    k_energy_stage<1><<<grid, 256, 0, st>>>(R, T, T, S.ws.rows, T1);
    k_energy_stage<2><<<grid, 256, 0, st>>>(R, T1, T, S.ws.rows, T);
    e = cudaGetLastError();
  }
  return e;
}
