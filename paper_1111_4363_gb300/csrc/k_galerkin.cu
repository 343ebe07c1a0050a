// Galerkin coarse operators (Sec. III, P A P^T with P^T = I): the spatial factors of the
// Kronecker normal operator, Sigma^{l+1}_kk' = I^T Sigma^l_kk' I, as radius-2 box stencils.
// They depend only on the static potential and the grid, so they are built once per
// la_set_hamiltonian; the per-step time factors Theta_kk' are combined with them later.
//
// The interpolation is a Kronecker product of 1D interpolations, and H = T_x + T_y + T_z + D with T_a the
// off-diagonal part of the 1D second difference and D = diag(dsum + V0).  So
//   I, X, X^2                 are products of 1D Galerkin tables on every level;
//   H    = sum T_a + D,
//   H^2  = sum T_a^2 + 2 sum_{a<b} T_a T_b + sum (T_a D + D T_a) + D^2,
//   H X  = sum T_a X + D X    are products of 1D tables plus terms linear in values of D at grid points;
//   X H  = (H X)^T,
// which the first coarse level contracts axis by axis, and the further levels contract axis by axis
// (z, y, x) from the previous level's stencils for the three products H, H^2, H X that are not Kronecker
// products.  All levels of a 96^3 grid: 4.5 ms (first 2.04, second 1.92, third 0.39); summing every fine pair
// of the two supports for every entry took 724 ms (645 + 70 + 9), bound by FP64 issue.
#include "la_internal.cuh"

namespace la {

// 1D Galerkin tables of one level: entry (type, axis, J, o) is (P^T S P)[J, J + o - 2] for the 1D operator S
// of the type, P the composite 1D interpolation to the level.  Types: I, T (off-diagonal second
// difference), T^2, and on the laser axis x, x^2, T x (zero on the other axes).
constexpr int kGalTypes = 6;
enum { kGalA = 0, kGalT = 1, kGalT2 = 2, kGalX = 3, kGalX2 = 4, kGalTX = 5 };

// Offset of (type, axis) in a level's table: the axes' points one after another, five offsets each.
__host__ __device__ __forceinline__ long long gal_tab(const int n[3], int type, int axis) {
  const long long tot = (long long)n[0] + n[1] + n[2];
  long long at = type * tot;
  if (axis > 0) at += n[0];
  if (axis > 1) at += n[1];
  return 5 * at;
}
long long galerkin_table_doubles(const int n[3]) { return 5LL * kGalTypes * ((long long)n[0] + n[1] + n[2]); }

// Weight of child i (0..3) of a coarse point: fine points 2J-1 .. 2J+2 with 1/4, 3/4, 3/4, 1/4 (transpose
// of the cell-centred linear interpolation).
__device__ __forceinline__ double gal_w(int i) { return (i == 1 || i == 2) ? 0.75 : 0.25; }
// the same as a function of the fine point a, zero outside the support or the grid
__device__ __forceinline__ double gal_wa(int a, int J, int nf) {
  const int i = a - (2 * J - 1);
  return (a < 0 || a >= nf || i < 0 || i > 3) ? 0.0 : gal_w(i);
}

// Entry (a, b) of the finest 1D operator of a type along axis `ax`.
__device__ __forceinline__ double gal_fine_1d(const FineOp& g, int type, int ax, int a, int b) {
  const int d = a > b ? a - b : b - a;
  const double h = ax == 0 ? g.h[0] : (ax == 1 ? g.h[1] : g.h[2]), ih2 = ax == 0 ? g.ih2[0] : (ax == 1 ? g.ih2[1] : g.ih2[2]);
  const double x0 = ax == 0 ? g.x0[0] : (ax == 1 ? g.x0[1] : g.x0[2]);
  const int n = ax == 0 ? g.n[0] : (ax == 1 ? g.n[1] : g.n[2]);
  const double w = -0.5 * ih2, xb = x0 + b * h;
  if (type >= kGalX && ax != g.lax) return 0.0;
  switch (type) {
    case kGalA: return d == 0 ? 1.0 : 0.0;
    case kGalT: return d == 1 ? w : 0.0;
    case kGalT2: return d == 0 ? w * w * ((a > 0 ? 1 : 0) + (a + 1 < n ? 1 : 0)) : (d == 2 ? w * w : 0.0);
    case kGalX: return d == 0 ? xb : 0.0;
    case kGalX2: return d == 0 ? xb * xb : 0.0;
    default: return d == 1 ? w * xb : 0.0;
  }
}

// Whether the finest 1D operator of a type has an entry at distance d.
__device__ __forceinline__ bool gal_nonzero(int type, int d) {
  if (type == kGalT || type == kGalTX) return d == 1 || d == -1;
  return d == 0 || (type == kGalT2 && (d == 2 || d == -2));
}

// One thread per table entry; nf, nc the points per axis of the finer level and of this one.
template <bool FROM_FINE>
__global__ void k_gal_1d(FineOp g, int3 nf3, int3 nc3, const double* __restrict__ tf, double* __restrict__ tc) {
  const int nf[3] = {nf3.x, nf3.y, nf3.z}, nc[3] = {nc3.x, nc3.y, nc3.z};
  const long long tot = (long long)nc[0] + nc[1] + nc[2];
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 5 * kGalTypes * tot) return;
  const int o = (int)(t % 5) - 2;
  const long long r = t / 5;
  const int type = (int)(r / tot);
  int J = (int)(r % tot), ax = 0;
  if (J >= nc[0]) { J -= nc[0]; ax = 1; }
  if (ax == 1 && J >= nc[1]) { J -= nc[1]; ax = 2; }
  const int nfa = ax == 0 ? nf[0] : (ax == 1 ? nf[1] : nf[2]), nca = ax == 0 ? nc[0] : (ax == 1 ? nc[1] : nc[2]);
  double s = 0.0;
  if (ax >= g.dim) {
    s = (type == kGalA && o == 0) ? 1.0 : 0.0;
  } else if (J + o >= 0 && J + o < nca) {
    const int K = J + o;
    const double* f = FROM_FINE ? nullptr : tf + gal_tab(nf, type, ax);
    for (int i = 0; i < 4; ++i) {
      const int a = 2 * J - 1 + i;
      if (a < 0 || a >= nfa) continue;
      for (int j = 0; j < 4; ++j) {
        const int b = 2 * K - 1 + j;
        if (b < 0 || b >= nfa || b - a > 2 || a - b > 2) continue;
        // most of the pairs, which cost the most on a long 1D grid: 343 -> 217 us a call on 100,352 points, two levels
        if (FROM_FINE && !gal_nonzero(type, b - a)) continue;
        s += gal_w(i) * gal_w(j) * (FROM_FINE ? gal_fine_1d(g, type, ax, a, b) : f[5LL * a + (b - a + 2)]);
      }
    }
  }
  tc[t] = s;
}

// Entry (J, o) of the three factors that are Kronecker products on every level: I, X (pairs (0,2) and
// (2,0)) and X^2.
__device__ __forceinline__ void gal_write_sep(double* __restrict__ s, int nbox, double sI, double sX, double sX2) {
  s[0] = sI;
  s[2 * nbox] = sX;
  s[6 * nbox] = sX;
  s[8 * nbox] = sX2;
}

// I, X and X^2 of the levels after the first, one thread per (coarse point J, offset o).
__global__ void __launch_bounds__(128) k_gal_sep(int lax, LevelGeom C, const double* __restrict__ tab,
                                                 double* __restrict__ sc) {
  const int nbox = box5_count(C.dim);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)C.np * nbox) return;
  const int J = (int)(t / nbox), o = (int)(t - (long long)J * nbox);
  const int ox = o % 5 - 2, oy = C.dim > 1 ? (o / 5) % 5 - 2 : 0, oz = C.dim > 2 ? o / 25 - 2 : 0;
  const int jx = J % C.n[0], jr = J / C.n[0], jy = jr % C.n[1], jz = jr / C.n[1];
  const int nc[3] = {C.n[0], C.n[1], C.n[2]};
  const long long ex = 5LL * jx + ox + 2, ey = 5LL * jy + oy + 2, ez = 5LL * jz + oz + 2;
  const double ax = tab[gal_tab(nc, kGalA, 0) + ex], ay = tab[gal_tab(nc, kGalA, 1) + ey],
               az = tab[gal_tab(nc, kGalA, 2) + ez];
  const long long el = lax == 0 ? ex : (lax == 1 ? ey : ez);
  const double x1 = tab[gal_tab(nc, kGalX, lax) + el], x2 = tab[gal_tab(nc, kGalX2, lax) + el];
  const double rest = lax == 0 ? ay * az : (lax == 1 ? ax * az : ax * ay);
  gal_write_sep(sc + sigma_offset(J, 0, o, nbox), nbox, ax * ay * az, x1 * rest, x2 * rest);
}

// First coarse level, all nine factors: one CTA per chunk of kGalChunk coarse points along x of one row
// (Jy, Jz).  The terms in D are contracted axis by axis.  With w_J the interpolation weights of J, the two
// forms of one axis are
//   W(c) = w_J(c) w_K(c)                                               (D and its powers),
//   G(c) = t (w_J(c) (w_K(c-1) + w_K(c+1)) + w_K(c) (w_J(c-1) + w_J(c+1)))    (T_a D + D T_a),
// nonzero for the six fine points 2J-2 .. 2J+3, and per entry
//   H += W W W D,  H X += W W W (D x),  H^2 += W W W D^2 + (G W W + W G W + W W G) D.
// z is contracted first, then y, for the fine x of the chunk all at once; the last step sums over x and
// adds the products of the 1D tables: about 1000 + 125 x 40 FP64 operations per coarse point.  The
// same sums taken per entry over the 4^3 points took 21.5 ms on 96^3, bound by FP64 issue with most lanes idle.
// In 1D a point has 5 entries only, so a CTA takes 64 points: 343 us instead of 349 us a call on 100,352 points.
constexpr int kGalChunk = 8, kGalChunk1D = 64, kGalThreads = 128;

// W and G of coarse point J and offset o on one axis at fine point c (zero where c or J + o is outside).
__device__ __forceinline__ void gal_wg(int J, int o, int c, int nf, int nc, double t, double& W, double& G) {
  const int K = J + o;
  W = G = 0.0;
  if (K < 0 || K >= nc || c < 0 || c >= nf) return;
  const double a = gal_wa(c, J, nf), b = gal_wa(c, K, nf);
  W = a * b;
  G = t * (a * (gal_wa(c - 1, K, nf) + gal_wa(c + 1, K, nf)) + b * (gal_wa(c - 1, J, nf) + gal_wa(c + 1, J, nf)));
}

template <int DIM>
__global__ void __launch_bounds__(kGalThreads) k_gal_first(FineOp g, LevelGeom C, const double* __restrict__ tab,
                                                           double* __restrict__ sc) {
  constexpr int OY = DIM > 1 ? 5 : 1, OZ = DIM > 2 ? 5 : 1, NBOX = 5 * OY * OZ;
  constexpr int RY = DIM > 1 ? 6 : 1, RZ = DIM > 2 ? 6 : 1;   // fine rows per axis
  constexpr int CY = DIM > 1 ? 2 : 0, CZ = DIM > 2 ? 2 : 0;   // index of offset 0
  constexpr int NJ = DIM > 1 ? kGalChunk : kGalChunk1D, NX = 2 * NJ + 4;   // coarse points and fine x of a chunk
  __shared__ double F[3][NX][RZ][RY];        // D, D^2, D x
  __shared__ double ZW[3][NX][RY][OZ];       // contracted over z with W
  __shared__ double ZG[NX][RY][OZ];          // D contracted with G
  __shared__ double YW[3][NX][OZ][OY];       // then over y with W
  __shared__ double YG[NX][OZ][OY];          // G W + W G of D
  __shared__ double wx[NJ][5][6], gx[NJ][5][6], wy[OY][RY], gy[OY][RY], wz[OZ][RZ], gz[OZ][RZ];
  const int tid = threadIdx.x;
  const int nchunk = (C.n[0] + NJ - 1) / NJ;
  const int ch = blockIdx.x % nchunk, row = blockIdx.x / nchunk;
  const int jy = row % C.n[1], jz = row / C.n[1];
  const int J0 = ch * NJ, nj = min(NJ, C.n[0] - J0);
  const int fx0 = 2 * J0 - 2, fy0 = DIM > 1 ? 2 * jy - 2 : 0, fz0 = DIM > 2 ? 2 * jz - 2 : 0;
  for (int t = tid; t < nj * 30; t += kGalThreads) {
    const int j = t / 30, o = (t / 6) % 5, i = t % 6;
    gal_wg(J0 + j, o - 2, 2 * (J0 + j) - 2 + i, g.n[0], C.n[0], -0.5 * g.ih2[0], wx[j][o][i], gx[j][o][i]);
  }
  if (DIM > 1) {
    for (int t = tid; t < OY * RY; t += kGalThreads)
      gal_wg(jy, t / RY - 2, fy0 + t % RY, g.n[1], C.n[1], -0.5 * g.ih2[1], wy[t / RY][t % RY], gy[t / RY][t % RY]);
  } else if (tid == 0) {
    wy[0][0] = 1.0;
    gy[0][0] = 0.0;
  }
  if (DIM > 2) {
    for (int t = tid; t < OZ * RZ; t += kGalThreads)
      gal_wg(jz, t / RZ - 2, fz0 + t % RZ, g.n[2], C.n[2], -0.5 * g.ih2[2], wz[t / RZ][t % RZ], gz[t / RZ][t % RZ]);
  } else if (tid == 0) {
    wz[0][0] = 1.0;
    gz[0][0] = 0.0;
  }
  for (int t = tid; t < RZ * RY * NX; t += kGalThreads) {
    const int lx = t % NX, ly = (t / NX) % RY, lz = t / (NX * RY);
    const int x = fx0 + lx, y = fy0 + ly, z = fz0 + lz;
    double d = 0.0, xl = 0.0;
    if (fine_in(g, x, y, z)) {
      d = g.dsum + g.V0[(z * g.n[1] + y) * g.n[0] + x];
      xl = fine_x(g, x, y, z);
    }
    F[0][lx][lz][ly] = d;
    F[1][lx][lz][ly] = d * d;
    F[2][lx][lz][ly] = d * xl;
  }
  __syncthreads();
  for (int t = tid; t < NX * RY * OZ; t += kGalThreads) {
    const int oz = t % OZ, ly = (t / OZ) % RY, lx = t / (OZ * RY);
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, ag = 0.0;
#pragma unroll
    for (int i = 0; i < RZ; ++i) {
      const double w = wz[oz][i], d = F[0][lx][i][ly];
      a0 = fma(w, d, a0);
      a1 = fma(w, F[1][lx][i][ly], a1);
      a2 = fma(w, F[2][lx][i][ly], a2);
      ag = fma(gz[oz][i], d, ag);
    }
    ZW[0][lx][ly][oz] = a0;
    ZW[1][lx][ly][oz] = a1;
    ZW[2][lx][ly][oz] = a2;
    ZG[lx][ly][oz] = ag;
  }
  __syncthreads();
  for (int t = tid; t < NX * OZ * OY; t += kGalThreads) {
    const int oy = t % OY, oz = (t / OY) % OZ, lx = t / (OY * OZ);
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, ag = 0.0;
#pragma unroll
    for (int i = 0; i < RY; ++i) {
      const double w = wy[oy][i], d = ZW[0][lx][i][oz];
      a0 = fma(w, d, a0);
      a1 = fma(w, ZW[1][lx][i][oz], a1);
      a2 = fma(w, ZW[2][lx][i][oz], a2);
      ag = fma(gy[oy][i], d, ag);
      ag = fma(w, ZG[lx][i][oz], ag);
    }
    YW[0][lx][oz][oy] = a0;
    YW[1][lx][oz][oy] = a1;
    YW[2][lx][oz][oy] = a2;
    YG[lx][oz][oy] = ag;
  }
  __syncthreads();
  const int nc[3] = {C.n[0], C.n[1], C.n[2]};
  const double* tA[3] = {tab + gal_tab(nc, kGalA, 0), tab + gal_tab(nc, kGalA, 1), tab + gal_tab(nc, kGalA, 2)};
  const double* tT[3] = {tab + gal_tab(nc, kGalT, 0), tab + gal_tab(nc, kGalT, 1), tab + gal_tab(nc, kGalT, 2)};
  const double* tS[3] = {tab + gal_tab(nc, kGalT2, 0), tab + gal_tab(nc, kGalT2, 1), tab + gal_tab(nc, kGalT2, 2)};
  const double *tX = tab + gal_tab(nc, kGalX, g.lax), *tX2 = tab + gal_tab(nc, kGalX2, g.lax),
               *tTX = tab + gal_tab(nc, kGalTX, g.lax);
  for (int t = tid; t < nj * NBOX; t += kGalThreads) {
    const int j = t / NBOX, e = t - j * NBOX;
    const int oxi = e % 5, oyi = (e / 5) % OY, ozi = e / (5 * OY);
    const int jx = J0 + j, kx = jx + oxi - 2, ky = jy + oyi - CY, kz = jz + ozi - CZ;
    const bool kin = kx >= 0 && kx < C.n[0] && ky >= 0 && ky < C.n[1] && kz >= 0 && kz < C.n[2];
    // table entries of offset o: index o + 2 on every axis (unused axes hold offset 0 there)
    const long long ex = 5LL * jx + oxi, ey = 5LL * jy + oyi - CY + 2, ez = 5LL * jz + ozi - CZ + 2;
    const double ax = tA[0][ex], ay = tA[1][ey], az = tA[2][ez];
    const double hx = tT[0][ex], hy = tT[1][ey], hz = tT[2][ez];
    const double ayz = ay * az, hyz = fma(hy, az, ay * hz);
    const double H0 = fma(hx, ayz, ax * hyz);
    double H2 = fma(2.0 * hx, hyz, tS[0][ex] * ayz);
    H2 = fma(ax, fma(tS[1][ey], az, fma(ay, tS[2][ez], 2.0 * hy * hz)), H2);
    double H = H0, HX, sX, sX2;
    if (g.lax == 0) {
      HX = fma(tTX[ex], ayz, tX[ex] * hyz);
      sX = tX[ex] * ayz;
      sX2 = tX2[ex] * ayz;
    } else {
      const long long el = g.lax == 1 ? ey : ez;
      const double ao = g.lax == 1 ? az : ay, ho = g.lax == 1 ? hz : hy;   // the other of y and z
      HX = fma(tTX[el], ax * ao, tX[el] * fma(hx, ao, ax * ho));
      sX = tX[el] * (ax * ao);
      sX2 = tX2[el] * (ax * ao);
    }
    if (kin)
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        const int lx = 2 * j + i;
        const double w = wx[j][oxi][i], yd = YW[0][lx][ozi][oyi];
        H = fma(w, yd, H);
        H2 = fma(w, YW[1][lx][ozi][oyi] + YG[lx][ozi][oyi], H2);
        H2 = fma(gx[j][oxi][i], yd, H2);
        HX = fma(w, YW[2][lx][ozi][oyi], HX);
      }
    const int J = (jz * C.n[1] + jy) * C.n[0] + jx;
    double* s = sc + sigma_offset(J, 0, e, NBOX);
    gal_write_sep(s, NBOX, kin ? ax * ayz : 0.0, kin ? sX : 0.0, kin ? sX2 : 0.0);
    s[NBOX] = s[3 * NBOX] = kin ? H : 0.0;
    s[4 * NBOX] = kin ? H2 : 0.0;
    s[5 * NBOX] = kin ? HX : 0.0;
    // X H = (H X)^T: to the transposed entry (K, -o), or this one's zero where K is outside
    sc[kin ? sigma_offset((kz * C.n[1] + ky) * C.n[0] + kx, 7, NBOX - 1 - e, NBOX) : sigma_offset(J, 7, e, NBOX)] =
        kin ? HX : 0.0;
  }
}

// Further levels in 2D and 3D, the factors (0,1), (1,1), (1,2) (and their copies (1,0) and (2,1)): one CTA per chunk of
// kGalChunk coarse points along x of one row (Jy, Jz) and one factor.  It walks the fine points of the row;
// the stencils of the 4 x 4 fine rows at one fine x are staged in shared memory (the next ones in flight),
// contracted over z and y (both the rows and the offsets), and every second fine x completes a coarse
// point from the last four contracted stencils: about 11,000 FMAs per coarse point and factor in 3D, against
// 8^3 x 125 x 4.6 for the direct double sum.  48^3 -> 24^3: 1.92 ms against 70 ms, bound by FP64 issue (0.9 ms of FMAs).
template <int DIM>
__global__ void __launch_bounds__(kGalThreads) k_gal_contract(LevelGeom F, const double* __restrict__ sf, LevelGeom C,
                                                              double* __restrict__ sc) {
  constexpr int OX = 5, OY = 5, OZ = DIM > 2 ? 5 : 1, NBOX = OX * OY * OZ;
  constexpr int AY = 4, AZ = DIM > 2 ? 4 : 1, NROW = AY * AZ;
  __shared__ double S[2][NROW * NBOX];
  __shared__ double Z[AY * NBOX];       // [ay][oz'][oy][ox]
  __shared__ double Y[4][NBOX];         // contracted over z and y, ring over the fine x
  const int tid = threadIdx.x;
  const int nchunk = (C.n[0] + kGalChunk - 1) / kGalChunk;
  const int ch = blockIdx.x % nchunk, row = blockIdx.x / nchunk;
  const int pair = blockIdx.y == 0 ? 1 : (blockIdx.y == 1 ? 4 : 5);
  const int jy = row % C.n[1], jz = row / C.n[1];
  const int J0 = ch * kGalChunk, J1 = min(J0 + kGalChunk, C.n[0]);
  auto fine_y = [&](int i) { return 2 * jy - 1 + i; };
  auto fine_z = [&](int i) { return DIM > 2 ? 2 * jz - 1 + i : jz; };
  auto stage = [&](int ax, double* dst) {
    if (ax >= 0 && ax < F.n[0])
      for (int t = tid; t < NROW * NBOX; t += kGalThreads) {
        const int r = t / NBOX, e = t - r * NBOX;
        const int fy = fine_y(r % AY), fz = fine_z(r / AY);
        if (fy >= 0 && fy < F.n[1] && fz >= 0 && fz < F.n[2]) {
          const double* src = sf + sigma_offset((fz * F.n[1] + fy) * F.n[0] + ax, pair, e, NBOX);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst + t)), "l"(src) : "memory");
        } else {
          dst[t] = 0.0;   // rows outside the grid carry no weight
        }
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int a0 = 2 * J0 - 1, a1 = 2 * (J1 - 1) + 2;
  stage(a0, S[0]);
  for (int ax = a0; ax <= a1; ++ax) {
    const double* Sx = S[(ax - a0) & 1];
    if (ax < a1) {
      stage(ax + 1, S[(ax + 1 - a0) & 1]);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const bool in = ax >= 0 && ax < F.n[0];
    if (in) {
      // z: Z[ay][oz'] = sum over fine z of the row (i) and of the offset's row (j)
      for (int t = tid; t < AY * NBOX; t += kGalThreads) {
        const int ay = t / NBOX, e = t - ay * NBOX, oxy = e % (OX * OY), ozc = e / (OX * OY) - (DIM > 2 ? 2 : 0);
        double v = 0.0;
        if (DIM > 2) {
          const int kz = jz + ozc;
          if (kz >= 0 && kz < C.n[2])
#pragma unroll
            for (int i = 0; i < AZ; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int d = 2 * ozc + j - i, b = 2 * kz - 1 + j;
                if (d >= -2 && d <= 2 && b >= 0 && b < F.n[2])
                  v = fma(gal_w(i) * gal_w(j), Sx[(i * AY + ay) * NBOX + (d + 2) * (OX * OY) + oxy], v);
              }
        } else {
          v = Sx[ay * NBOX + e];
        }
        Z[t] = v;
      }
    }
    __syncthreads();
    if (in) {
      // y: contracted over the fine y rows
      for (int e = tid; e < NBOX; e += kGalThreads) {
        const int ox = e % OX, oyc = (e / OX) % OY - 2, oz = e / (OX * OY);
        double v = 0.0;
        const int ky = jy + oyc;
        if (ky >= 0 && ky < C.n[1])
#pragma unroll
          for (int i = 0; i < AY; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int d = 2 * oyc + j - i, b = 2 * ky - 1 + j;
              if (d >= -2 && d <= 2 && b >= 0 && b < F.n[1])
                v = fma(gal_w(i) * gal_w(j), Z[i * NBOX + (oz * OY + (d + 2)) * OX + ox], v);
            }
        Y[ax & 3][e] = v;
      }
    }
    __syncthreads();
    // x: fine x = 2 J + 2 completes coarse point J
    if (!(ax & 1) && ax >= 2 * J0 + 2) {
      const int jx = (ax - 2) >> 1;
      for (int e = tid; e < NBOX; e += kGalThreads) {
        const int ox = e % OX - 2, oyi = (e / OX) % OY, ozi = e / (OX * OY);
        const int kx = jx + ox, ky = jy + oyi - 2, kz = jz + (DIM > 2 ? ozi - 2 : 0);
        const bool kin = kx >= 0 && kx < C.n[0] && ky >= 0 && ky < C.n[1] && kz >= 0 && kz < C.n[2];
        double v = 0.0;
        if (kin)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int a = 2 * jx - 1 + i, b = 2 * kx - 1 + j, d = 2 * ox + j - i;
              if (d >= -2 && d <= 2 && a >= 0 && a < F.n[0] && b >= 0 && b < F.n[0])
                v = fma(gal_w(i) * gal_w(j), Y[a & 3][(e - e % OX) + d + 2], v);
            }
        const int J = (jz * C.n[1] + jy) * C.n[0] + jx;
        sc[sigma_offset(J, pair, e, NBOX)] = v;
        if (pair == 1) sc[sigma_offset(J, 3, e, NBOX)] = v;
        if (pair == 5)   // X H = (H X)^T; rows of entries outside the grid are zero
          sc[kin ? sigma_offset((kz * C.n[1] + ky) * C.n[0] + kx, 7, NBOX - 1 - e, NBOX)
                 : sigma_offset(J, 7, e, NBOX)] = v;
      }
    }
  }
}

// The same in 1D, one thread per entry: 16 products at most, so nothing is gained by contracting (a level of 25,088
// points adds 48 us to a call, 118 us with the walk along x).
__global__ void __launch_bounds__(128) k_gal_line(LevelGeom F, const double* __restrict__ sf, LevelGeom C,
                                                  double* __restrict__ sc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 5 * C.np) return;
  const int pair = blockIdx.y == 0 ? 1 : (blockIdx.y == 1 ? 4 : 5);
  const int J = t / 5, e = t - 5 * J, K = J + e - 2;
  const bool kin = K >= 0 && K < C.np;
  double v = 0.0;
  if (kin)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int a = 2 * J - 1 + i, b = 2 * K - 1 + j, d = b - a;
        if (d >= -2 && d <= 2 && a >= 0 && a < F.np && b >= 0 && b < F.np)
          v = fma(gal_w(i) * gal_w(j), sf[sigma_offset(a, pair, d + 2, 5)], v);
      }
  sc[sigma_offset(J, pair, e, 5)] = v;
  if (pair == 1) sc[sigma_offset(J, 3, e, 5)] = v;
  if (pair == 5) sc[kin ? sigma_offset(K, 7, 4 - e, 5) : sigma_offset(J, 7, e, 5)] = v;
}

void launch_galerkin(const FineOp& g, const LevelGeom* geo, int levels, double* const* sigma, double* tab0,
                     double* tab1, cudaStream_t s) {
  double* tab[2] = {tab0, tab1};
  for (int l = 1; l < levels; ++l) {
    const LevelGeom &F = geo[l - 1], &C = geo[l];
    const int3 nf = make_int3(F.n[0], F.n[1], F.n[2]), nc = make_int3(C.n[0], C.n[1], C.n[2]);
    const long long nt = galerkin_table_doubles(C.n), ne = (long long)C.np * box5_count(C.dim);
    const unsigned tb = (unsigned)((nt + 127) / 128), eb = (unsigned)((ne + 127) / 128);
    if (l == 1) {
      k_gal_1d<true><<<tb, 128, 0, s>>>(g, nf, nc, nullptr, tab[1]);
      const int nj = C.dim == 1 ? kGalChunk1D : kGalChunk;
      const unsigned grid = (unsigned)(((C.n[0] + nj - 1) / nj) * C.n[1] * C.n[2]);
      if (C.dim == 1) k_gal_first<1><<<grid, kGalThreads, 0, s>>>(g, C, tab[1], sigma[1]);
      else if (C.dim == 2) k_gal_first<2><<<grid, kGalThreads, 0, s>>>(g, C, tab[1], sigma[1]);
      else k_gal_first<3><<<grid, kGalThreads, 0, s>>>(g, C, tab[1], sigma[1]);
    } else {
      k_gal_1d<false><<<tb, 128, 0, s>>>(g, nf, nc, tab[(l - 1) & 1], tab[l & 1]);
      k_gal_sep<<<eb, 128, 0, s>>>(g.lax, C, tab[l & 1], sigma[l]);
      const dim3 grid((unsigned)(((C.n[0] + kGalChunk - 1) / kGalChunk) * C.n[1] * C.n[2]), 3);
      if (C.dim == 1) k_gal_line<<<dim3((unsigned)((5LL * C.np + 127) / 128), 3), 128, 0, s>>>(F, sigma[l - 1], C, sigma[l]);
      else if (C.dim == 2) k_gal_contract<2><<<grid, kGalThreads, 0, s>>>(F, sigma[l - 1], C, sigma[l]);
      else k_gal_contract<3><<<grid, kGalThreads, 0, s>>>(F, sigma[l - 1], C, sigma[l]);
    }
  }
}

}  // namespace la
