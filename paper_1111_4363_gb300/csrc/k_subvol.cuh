// Subvolume relaxation kernels (Sec. II), templated on the arithmetic type R (double or float).
//
// A subvolume U is a block of grid points with all K time functions: n = |U| K unknowns,
// padded to NPAD (multiple of 16) with identity rows.  Its local least-squares problem
// (minimise the residual norm N over c_U, everything else fixed) has the Hermitian
// positive-definite matrix G_UU = sum_kk' Sigma_kk'[U, U] (x) Theta_kk' and right-hand side
// (M~^dagger Wt r)_U (finest level) or (g - G e)_U (Galerkin levels).
//
// Factor store of one subvolume: lower Cholesky factor L of G_UU in 16 x 16 blocks, block rows
// I = 0..NB-1 and block columns J <= I in the order (0,0), (1,0), (1,1), (2,0), ..., in one of three layouts:
// - block (I, I) holds inv(L_II) instead of L_II, so that every triangular-solve step is a mat-vec (FP64, and
//   complex64 from 33 unknowns on but for the next);
// - complex64 of more than 128 unknowns with a band of at most 8 blocks (factor_is_super): the 4 x 4 blocks of each
//   diagonal superblock hold the inverse of L's superblock;
// - complex64 of at most 32 unknowns (factor_is_inverse): the record holds inv(L) whole.
// The inverses keep the 32 bits of the factors they replace; the bound of a solve with them has one more factor of the
// block's condition number.  Errors of a coloured pass against the same pass in FP64 over those of substitution,
// geometric means over shapes, K and states: inv(L) 0.87, 0.92 and 0.98 (weights 0, 2 and 1), the superblocks 1.04,
// 1.10 and 1.25.
#pragma once
#include "la_internal.cuh"

namespace la {

template <typename CT> struct Re;
template <> struct Re<double2> { typedef double T; };
template <> struct Re<float2> { typedef float T; };

template <typename CT> __device__ __forceinline__ CT mkc(typename Re<CT>::T a, typename Re<CT>::T b) {
  CT r; r.x = a; r.y = b; return r;
}
// acc += a * b
template <typename CT> __device__ __forceinline__ void cfma(CT& acc, const CT a, const CT b) {
  acc.x = fma(a.x, b.x, acc.x); acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y); acc.y = fma(a.y, b.x, acc.y);
}
// acc += conj(a) * b
template <typename CT> __device__ __forceinline__ void cfma_conj(CT& acc, const CT a, const CT b) {
  acc.x = fma(a.x, b.x, acc.x); acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y); acc.y = fma(-a.y, b.x, acc.y);
}

// a -= x conj(y)
template <typename CT> __device__ __forceinline__ void sub_conj(CT& a, const CT x, const CT y) {
  a.x = fma(-x.x, y.x, a.x); a.x = fma(-x.y, y.y, a.x);
  a.y = fma(-x.y, y.x, a.y); a.y = fma(x.x, y.y, a.y);
}

constexpr int kFactorThreads = 256;
constexpr int kSweepThreads = 128;
constexpr int kSuperThreads = 256;   // sweeps with superblock factors

__device__ __forceinline__ void local_coords(int i, const int e[3], int& x, int& y, int& z) {
  x = i % e[0];
  int r = i / e[0];
  y = r % e[1];
  z = r / e[1];
}

// ======================================================================== factorisation
// One 256-thread CTA per subvolume of a level; two CTAs per SM.  The padded matrix lives in
// shared memory as a packed lower triangle (assembled tile-cyclically: thread (tid/16, tid%16)
// writes entries (16 I + tid/16, 16 J + tid%16)).  Right-looking Cholesky with two barriers per
// pair of columns: (A) the columns are scaled and published, (B) the trailing triangle takes both
// with its entries spread linearly over the threads; one thread updates the next two pivots first
// and computes their reciprocal square roots while the others are still updating (lookahead), so
// the pivot chain is off the critical path.
__host__ __device__ constexpr int tri_index(int r, int c) { return r * (r + 1) / 2 + c; }

// Small matrices leave most threads of a CTA idle in the later columns, so a CTA factorises
// factor_mpc(NPAD) matrices together: each phase's work is split over the entries of all of them and
// they share the two barriers per column.
__host__ __device__ constexpr int factor_mpc(int npad) { return npad <= 32 ? 8 : (npad <= 64 ? 2 : 1); }

// Bytes of one matrix's pair table, whose place holds a column of the factorisation later.
__host__ __device__ constexpr size_t factor_pair_bytes(int npair, int npad, size_t csize) {
  const size_t p = sizeof(double) * (size_t)npair * LA_NPAIR, c = csize * (size_t)npad;
  return p > c ? p : c;
}

template <typename R, int NPAD, int MPC>
__global__ void __launch_bounds__(kFactorThreads, 2)
k_factor(LevelGeom L, FineOp g, int is_fine, int nptsmax, const R* __restrict__ sigma,
         const TimeMats* __restrict__ tm, typename C2<R>::T* __restrict__ factors, int* __restrict__ status) {
  typedef typename C2<R>::T CT;
  constexpr int NTRI = NPAD * (NPAD + 1) / 2;
  constexpr int NB = NPAD / LA_BLK;
  extern __shared__ __align__(16) unsigned char smem[];
  const int K = tm->K, KK = K * K;
  const int npair_max = nptsmax * (nptsmax + 1) / 2;
  CT* sA = reinterpret_cast<CT*>(smem);                       // [MPC][NTRI] packed lower triangles
  CT* sCol = sA + MPC * NTRI;                                 // [MPC][NPAD] scaled column j of the pair
  R* sInv = reinterpret_cast<R*>(sCol + MPC * NPAD);          // [MPC][NPAD] 1/L_jj
  double* sP = reinterpret_cast<double*>(sInv + MPC * NPAD);  // [9][K*K]
  double* sPair = sP + LA_NPAIR * LA_KMAX * LA_KMAX;          // [MPC][npair_max][9], point pairs i >= j
  int* sMask = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(sPair) +
                                      MPC * factor_pair_bytes(npair_max, NPAD, sizeof(CT)));  // [MPC][npair_max]
  CT* sCol1 = reinterpret_cast<CT*>(sPair);   // [MPC][NPAD] scaled column j + 1, in the pairs' place after the assembly

  const int tid = threadIdx.x, ti = tid >> 4, tk = tid & 15;
  // the CTA's matrices; slots past the last subvolume factorise an identity and store nothing
  int bsv[MPC], nn_[MPC], npts_[MPC];
  int o_[MPC][3], e_[MPC][3];
#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    bsv[mi] = blockIdx.x * MPC + mi;
    if (bsv[mi] < L.nsub) {
      subvol_box(L, bsv[mi], o_[mi], e_[mi]);
      npts_[mi] = e_[mi][0] * e_[mi][1] * e_[mi][2];
    } else {
      o_[mi][0] = o_[mi][1] = o_[mi][2] = 0;
      e_[mi][0] = e_[mi][1] = e_[mi][2] = 1;
      npts_[mi] = 0;
    }
    nn_[mi] = npts_[mi] * K;
  }

  for (int i = tid; i < LA_NPAIR * KK; i += kFactorThreads) sP[i] = tm->P[i / KK][i % KK];
  // pair tables for point pairs i >= j: the nine spatial factors Sigma_kk'[p_i, p_j] and a bit mask
  // of the nonzero ones (most pairs of a subvolume are too far apart for most factors)
  const int nbox = box5_count(L.dim);
  for (int t = tid; t < MPC * npair_max; t += kFactorThreads) {
    const int mi = t / npair_max, q = t - mi * npair_max;
    int npts = 0, o[3] = {0, 0, 0}, e[3] = {1, 1, 1};
#pragma unroll
    for (int u = 0; u < MPC; ++u)
      if (u == mi) {
        npts = npts_[u];
        for (int a = 0; a < 3; ++a) { o[a] = o_[u][a]; e[a] = e_[u][a]; }
      }
    if (q >= npts * (npts + 1) / 2) continue;
    int i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > q) --i;
    while ((i + 1) * (i + 2) / 2 <= q) ++i;
    const int j = q - i * (i + 1) / 2;
    int ix, iy, iz, jx, jy, jz;
    local_coords(i, e, ix, iy, iz);
    local_coords(j, e, jx, jy, jz);
    const int px = o[0] + ix, py = o[1] + iy, pz = o[2] + iz;
    const int qx = o[0] + jx, qy = o[1] + jy, qz = o[2] + jz;
    double s9[LA_NPAIR];
    if (is_fine) {
      fine_sigma(g, px, py, pz, qx, qy, qz, s9);
    } else {
      const int dx = qx - px, dy = qy - py, dz = qz - pz;
      const bool near = abs(dx) <= 2 && abs(dy) <= 2 && abs(dz) <= 2;
      const int p = (pz * L.n[1] + py) * L.n[0] + px;
      const int ofs = near ? box5_index(L.dim, dx, dy, dz) : 0;
      for (int k = 0; k < LA_NPAIR; ++k) s9[k] = near ? sigma[sigma_offset(p, k, ofs, nbox)] : 0.0;
    }
    int mask = 0;
    double* dst = sPair + ((size_t)mi * npair_max + q) * LA_NPAIR;
    for (int k = 0; k < LA_NPAIR; ++k) {
      dst[k] = s9[k];
      if (s9[k] != 0.0) mask |= 1 << k;
    }
    sMask[mi * npair_max + q] = mask;
  }
  // padding rows: identity
  for (int t = tid; t < MPC * NTRI; t += kFactorThreads) {
    const int mi = t / NTRI, u = t - mi * NTRI;
    int r = (int)((sqrtf(8.0f * (float)u + 1.0f) - 1.0f) * 0.5f);
    while (r * (r + 1) / 2 > u) --r;
    while ((r + 1) * (r + 2) / 2 <= u) ++r;
    const int c = u - r * (r + 1) / 2;
    int n = 0;
#pragma unroll
    for (int w = 0; w < MPC; ++w) if (w == mi) n = nn_[w];
    if (r >= n) sA[t] = mkc<CT>((R)(r == c ? 1 : 0), (R)0);
  }
  __syncthreads();

  // ---- assemble pair-major: G_UU[(i,m),(j,n)] = sum_kk' Sigma_kk'[p_i, p_j] Theta_kk'[m, n].
  // Consecutive threads take the K*K entries of one point pair, so the skipped (zero) factors
  // are uniform across a warp except at pair boundaries.
  for (int t = tid; t < MPC * npair_max * KK; t += kFactorThreads) {
    const int mi = t / (npair_max * KK), tq = t - mi * npair_max * KK;
    const int q = tq / KK, mn = tq % KK, mm = mn / K, nn = mn % K;
    int npts = 0;
#pragma unroll
    for (int u = 0; u < MPC; ++u) if (u == mi) npts = npts_[u];
    if (q >= npts * (npts + 1) / 2) continue;
    int i = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > q) --i;
    while ((i + 1) * (i + 2) / 2 <= q) ++i;
    const int j = q - i * (i + 1) / 2;
    const int r = i * K + mm, c = j * K + nn;
    if (r < c) continue;
    const int mask = sMask[mi * npair_max + q];
    const double* pr = sPair + ((size_t)mi * npair_max + q) * LA_NPAIR;
    double re = 0.0, im = 0.0;
#pragma unroll
    for (int kk = 0; kk < LA_NPAIR; ++kk) {
      if (!((mask >> kk) & 1)) continue;
      const double v = pr[kk] * sP[kk * KK + mm * K + nn];
      const int ph = theta_phase(kk);
      if (ph == 0) re += v; else if (ph == 1) im += v; else im -= v;
    }
    sA[mi * NTRI + tri_index(r, c)] = mkc<CT>((R)re, (R)im);
  }
  __syncthreads();
  // ---- right-looking Cholesky, two columns at a time.  Work of each phase is spread linearly over exactly the
  // active entries of all the CTA's matrices (consecutive threads take consecutive entries of a row), so
  // every issued FP64 instruction has all lanes busy except in the last warp of a phase.
  // Columns j, j + 1 end at the last row that the point of j + 1 couples to (L.reach): the rows below stay exact
  // zeros in G and in the factor, so no phase visits them.  4x4 points x 6, 4096 matrices: 5.61 ms dense and one
  // column at a time, 4.18 ms with the zeros left out, 3.84 ms with two columns per pair of
  // barriers.
  // The pivots of columns j and j + 1 and the entry between them, by one thread per matrix.  c0, c1: the two columns
  // before, whose products are still to be subtracted (null for the first pair); they end at row `last`.
  auto pivots = [&](int mi, int j, const CT* c0, const CT* c1, int last) {
    CT* A = sA + mi * NTRI;
    const CT zero = mkc<CT>((R)0, (R)0);
    CT a00 = A[tri_index(j, j)], a10 = A[tri_index(j + 1, j)], a11 = A[tri_index(j + 1, j + 1)];
    if (c0) {
      const CT x0 = j <= last ? c0[j] : zero, x1 = j <= last ? c1[j] : zero;
      const CT y0 = j + 1 <= last ? c0[j + 1] : zero, y1 = j + 1 <= last ? c1[j + 1] : zero;
      sub_conj(a00, x0, x0); sub_conj(a00, x1, x1);
      sub_conj(a10, y0, x0); sub_conj(a10, y1, x1);
      sub_conj(a11, y0, y0); sub_conj(a11, y1, y1);
    }
    R d0 = a00.x;
    if (!(d0 > (R)0)) { atomicOr(status, 1); d0 = (R)1; }
    const R i0 = rsqrt(d0);
    const CT l = mkc<CT>(a10.x * i0, a10.y * i0);
    sub_conj(a11, l, l);
    R d1 = a11.x;
    if (!(d1 > (R)0)) { atomicOr(status, 1); d1 = (R)1; }
    const R i1 = rsqrt(d1);
    A[tri_index(j, j)] = mkc<CT>(d0 * i0, (R)0);
    A[tri_index(j + 1, j)] = l;
    A[tri_index(j + 1, j + 1)] = mkc<CT>(d1 * i1, (R)0);
    sInv[mi * NPAD + j] = i0;
    sInv[mi * NPAD + j + 1] = i1;
  };
  if (tid < MPC) pivots(tid, 0, nullptr, nullptr, 0);
  __syncthreads();
  for (int j = 0; j + 2 < NPAD; j += 2) {
    const int last = min(NPAD - 1, (fdiv(j + 1, L.fd_K) + L.reach + 1) * K - 1);
    const int rows = last - j - 1;   // rows j + 2 .. last
    // (A) columns j and j + 1, scaled and published
    for (int t = tid; t < MPC * rows; t += kFactorThreads) {
      const int mi = t / rows, r = j + 2 + (t - mi * rows);
      CT* A = sA + mi * NTRI;
      const R i0 = sInv[mi * NPAD + j], i1 = sInv[mi * NPAD + j + 1];
      CT v = A[tri_index(r, j)], w = A[tri_index(r, j + 1)];
      v.x *= i0; v.y *= i0;
      sub_conj(w, v, A[tri_index(j + 1, j)]);
      w.x *= i1; w.y *= i1;
      A[tri_index(r, j)] = v;
      A[tri_index(r, j + 1)] = w;
      sCol[mi * NPAD + r] = v;
      sCol1[mi * NPAD + r] = w;
    }
    __syncthreads();
    // (B) trailing update of the entries (r, c), j + 2 <= c <= r <= last; entry e of a trailing triangle lies in row
    // j + 1 + m with (m-1) m / 2 <= e < m (m+1) / 2.  The first three hold the next two pivots: one thread per
    // matrix updates them and takes the reciprocal square roots while the others go on (lookahead).
    if (tid < MPC) {
      pivots(tid, j + 2, sCol + tid * NPAD, sCol1 + tid * NPAD, last);
    }
    const int T = rows * (rows + 1) / 2 - 3;
    for (int t = kFactorThreads - 1 - tid; t < MPC * T; t += kFactorThreads) {
      const int mi = MPC > 1 ? t / T : 0, e = t - mi * T + 3;
      int m = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)e)) * 0.5f);
      while ((m - 1) * m / 2 > e) --m;
      while (m * (m + 1) / 2 <= e) ++m;
      const int r = j + 1 + m, c = j + 2 + (e - (m - 1) * m / 2);
      const CT* c0 = sCol + mi * NPAD;
      const CT* c1 = sCol1 + mi * NPAD;
      CT a = sA[mi * NTRI + tri_index(r, c)];
      sub_conj(a, c0[r], c0[c]);
      sub_conj(a, c1[r], c1[c]);
      sA[mi * NTRI + tri_index(r, c)] = a;
    }
    __syncthreads();
  }

  // ---- store: off-diagonal blocks as they are, diagonal blocks inverted
#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    if (bsv[mi] >= L.nsub) continue;
    CT* F = factors + (size_t)bsv[mi] * L.fsize;
    const CT* A = sA + mi * NTRI;
#pragma unroll
    for (int I = 1; I < NB; ++I)
#pragma unroll
      for (int J = 0; J < I; ++J)
        F[(size_t)(I * (I + 1) / 2 + J) * 256 + ti * LA_BLK + tk] = A[tri_index(LA_BLK * I + ti, LA_BLK * J + tk)];
  }
  // inv(L_II): thread (matrix, I, column jj) solves L_II x = e_jj by forward substitution
  if (tid < MPC * NB * LA_BLK) {
    const int mi = tid / (NB * LA_BLK), rem = tid - mi * NB * LA_BLK;
    const int I = rem / LA_BLK, jj = rem % LA_BLK, base = LA_BLK * I;
    int bm = 0;
#pragma unroll
    for (int u = 0; u < MPC; ++u) if (u == mi) bm = bsv[u];
    if (bm < L.nsub) {
      const CT* A = sA + mi * NTRI;
      const R* Inv = sInv + mi * NPAD;
      CT x[LA_BLK];
#pragma unroll
      for (int i = 0; i < LA_BLK; ++i) {
        CT acc = mkc<CT>(0, 0);
#pragma unroll
        for (int k = 0; k < i; ++k)
          if (k >= jj) cfma(acc, A[tri_index(base + i, base + k)], x[k]);
        const R rinv = Inv[base + i];
        if (i < jj) x[i] = mkc<CT>(0, 0);
        else if (i == jj) x[i] = mkc<CT>(rinv, (R)0);
        else x[i] = mkc<CT>(-acc.x * rinv, -acc.y * rinv);
      }
      CT* D = factors + (size_t)bm * L.fsize + (size_t)(I * (I + 1) / 2 + I) * 256;
#pragma unroll
      for (int i = 0; i < LA_BLK; ++i) D[i * LA_BLK + jj] = x[i];
    }
  }
}

// ------------------------------------------------------------------------ complex64 variant
// For complex64 the whole factor fits in registers: thread (ti, tk) keeps its tile-cyclic entries
// (16 I + ti, 16 J + tk), J <= I, in registers with compile-time tile indices.  Blocked
// right-looking Cholesky: the 16 columns of a panel are eliminated one by one inside the panel's
// block column only (two barriers per column, pivot lookahead), the finished panel goes to shared
// memory k-major, and every trailing block then takes one rank-16 update from it (row reads are
// broadcasts, column reads are consecutive), so the per-entry bookkeeping is paid once per 16
// columns instead of once per column.
// Matrices per CTA of the blocked factorisation: small ones share the column barriers (their
// per-thread register tiles stay small: NT = 6 complex for NPAD 48).  Up to 32 unknowns: k_factor_small.
__host__ __device__ constexpr int factor_c64_mpc(int npad) { return npad <= 48 ? 2 : 1; }

__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

// The blocked factorisation, written for a precision R; the mixed path runs it in complex64 (two
// CTAs per SM).  In complex128 its register tiles allow one CTA per SM, and measured slower than the
// shared-memory factorisation above (NPAD 96 at 256 x 256: 9.4 ms against 5.7 ms), so the FP64
// path does not use it.
template <typename R, int NPAD, int MPC>
__global__ void __launch_bounds__(kFactorThreads, sizeof(R) == 4 ? (NPAD <= 96 ? 3 : 2) : 1)
k_factor_blk(LevelGeom L, FineOp g, int is_fine, int nptsmax, const R* __restrict__ sigma,
             const TimeMats* __restrict__ tm, typename C2<R>::T* __restrict__ factors, int* __restrict__ status) {
  typedef typename C2<R>::T CT;
  constexpr int NB = NPAD / LA_BLK;
  constexpr int NT = NB * (NB + 1) / 2;
  extern __shared__ __align__(16) unsigned char smem[];
  const int K = tm->K, KK = K * K;
  const int nv = is_fine ? 2 : LA_NPAIR;
  const int pstride = nptsmax * nptsmax * nv;
  CT* sPan = reinterpret_cast<CT*>(smem);                          // [MPC][LA_BLK][NPAD] finished panel, k-major
  R* sInv = reinterpret_cast<R*>(sPan + MPC * LA_BLK * NPAD);     // [MPC][NPAD]
  CT* sDiag = reinterpret_cast<CT*>(sInv + MPC * NPAD);             // [MPC][NB][256]
  R* sP = reinterpret_cast<R*>(sDiag + MPC * NB * 256);             // [9][K*K]
  R* sPair = sP + LA_NPAIR * LA_KMAX * LA_KMAX;                     // [MPC][npts*npts][nv]
  R* sX = sPair + (size_t)MPC * pstride;                            // [MPC][npts] laser coordinate (finest)

  const int tid = threadIdx.x, ti = tid >> 4, tk = tid & 15;
  // the CTA's matrices; slots past the last subvolume factorise an identity and store nothing
  int bsv[MPC], npts_[MPC], o_[MPC][3], e_[MPC][3];
#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    bsv[mi] = blockIdx.x * MPC + mi;
    if (bsv[mi] < L.nsub) {
      subvol_box(L, bsv[mi], o_[mi], e_[mi]);
      npts_[mi] = e_[mi][0] * e_[mi][1] * e_[mi][2];
    } else {
      o_[mi][0] = o_[mi][1] = o_[mi][2] = 0;
      e_[mi][0] = e_[mi][1] = e_[mi][2] = 1;
      npts_[mi] = 0;
    }
  }
  for (int i = tid; i < LA_NPAIR * KK; i += kFactorThreads) sP[i] = (R)tm->P[i / KK][i % KK];
  for (int i = tid; i < MPC * NB * 256; i += kFactorThreads) sDiag[i] = mkc<CT>(0, 0);
  const int nbox = box5_count(L.dim);
#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    const int npts = npts_[mi];
    const int* o = o_[mi];
    const int* e = e_[mi];
    if (is_fine)
      for (int i = tid; i < npts; i += kFactorThreads) {
        int ix, iy, iz;
        local_coords(i, e, ix, iy, iz);
        sX[mi * nptsmax + i] = (R)fine_x(g, o[0] + ix, o[1] + iy, o[2] + iz);
      }
    for (int t = tid; t < npts * npts; t += kFactorThreads) {
      const int i = t / npts, j = t % npts;
      int ix, iy, iz, jx, jy, jz;
      local_coords(i, e, ix, iy, iz);
      local_coords(j, e, jx, jy, jz);
      const int px = o[0] + ix, py = o[1] + iy, pz = o[2] + iz;
      const int qx = o[0] + jx, qy = o[1] + jy, qz = o[2] + jz;
      R* dst = sPair + (size_t)mi * pstride + (size_t)t * nv;
      if (is_fine) {
        double s9[LA_NPAIR];
        fine_sigma(g, px, py, pz, qx, qy, qz, s9);
        dst[0] = (R)s9[1];
        dst[1] = (R)s9[4];
      } else {
        const int dx = qx - px, dy = qy - py, dz = qz - pz;
        const bool near = abs(dx) <= 2 && abs(dy) <= 2 && abs(dz) <= 2;
        const int p = (pz * L.n[1] + py) * L.n[0] + px;
        const int ofs = near ? box5_index(L.dim, dx, dy, dz) : 0;
        for (int k = 0; k < LA_NPAIR; ++k) dst[k] = near ? (R)sigma[sigma_offset(p, k, ofs, nbox)] : (R)0;
      }
    }
  }
  __syncthreads();

  CT a[MPC][NT];
#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    const int npts = npts_[mi], n = npts * K;
#pragma unroll
    for (int I = 0; I < NB; ++I) {
#pragma unroll
      for (int J = 0; J <= I; ++J) {
        const int r = LA_BLK * I + ti, c = LA_BLK * J + tk;
        // assembled in R (complex64: this factor only preconditions the FP64-refined iteration)
        R re = 0, im = 0;
        if (I == J && ti < tk) {
        } else if (r >= n || c >= n) {
          re = (r == c) ? (R)1 : (R)0;
        } else {
          const int i = r / K, mm = r % K, j = c / K, nn = c % K;
          R s9[LA_NPAIR];
          const R* pr = sPair + (size_t)mi * pstride + (size_t)(i * npts + j) * nv;
          if (is_fine) {
            const R xp = sX[mi * nptsmax + i], xq = sX[mi * nptsmax + j];
            const R same = (i == j) ? (R)1 : (R)0, Hpq = pr[0];
            s9[0] = same; s9[1] = Hpq; s9[2] = same * xp; s9[3] = Hpq; s9[4] = pr[1];
            s9[5] = Hpq * xq; s9[6] = same * xp; s9[7] = xp * Hpq; s9[8] = same * xp * xp;
          } else {
#pragma unroll
            for (int kk = 0; kk < LA_NPAIR; ++kk) s9[kk] = pr[kk];
          }
#pragma unroll
          for (int kk = 0; kk < LA_NPAIR; ++kk) {
            const R v = s9[kk] * sP[kk * KK + mm * K + nn];
            const int ph = theta_phase(kk);
            if (ph == 0) re += v; else if (ph == 1) im += v; else im -= v;
          }
        }
        a[mi][I * (I + 1) / 2 + J] = mkc<CT>(re, im);
      }
    }
  }
  if (tid == 0) {
#pragma unroll
    for (int mi = 0; mi < MPC; ++mi) {
      R d2 = a[mi][0].x;
      if (!(d2 > (R)0)) { atomicOr(status, 1); d2 = (R)1; }
      const R inv = rsq(d2);
      a[mi][0] = mkc<CT>(d2 * inv, 0);
      sInv[mi * NPAD] = inv;
    }
  }
  __syncthreads();

#pragma unroll
  for (int J0 = 0; J0 < NB; ++J0) {
    const int c0 = LA_BLK * J0 + tk;   // this thread's column inside the panel
    for (int jj = 0; jj < LA_BLK; ++jj) {
      const int j = LA_BLK * J0 + jj;
      // (A) owners of column j scale it and publish it
      if (tk == jj) {
#pragma unroll
        for (int mi = 0; mi < MPC; ++mi) {
          const R inv = sInv[mi * NPAD + j];
          CT* pan = sPan + (size_t)mi * LA_BLK * NPAD;
#pragma unroll
          for (int I = J0; I < NB; ++I) {
            const int r = LA_BLK * I + ti;
            if (r > j) {
              CT& v = a[mi][I * (I + 1) / 2 + J0];
              v.x *= inv;
              v.y *= inv;
              pan[jj * NPAD + r] = v;
            }
          }
        }
      }
      __syncthreads();
      if (jj == LA_BLK - 1) break;   // the panel's last column changes nothing inside the panel
      // (B) rank-1 update of the panel right of column j; the owner of entry (j+1, j+1) takes its rsqrt
      if (c0 > j) {
#pragma unroll
        for (int mi = 0; mi < MPC; ++mi) {
          const CT* pan = sPan + (size_t)mi * LA_BLK * NPAD;
          const CT y = pan[jj * NPAD + c0];
#pragma unroll
          for (int I = J0; I < NB; ++I) {
            const int r = LA_BLK * I + ti;
            if (r >= c0) {
              const CT xr = pan[jj * NPAD + r];
              CT& v = a[mi][I * (I + 1) / 2 + J0];
              v.x = fma(-xr.x, y.x, v.x); v.x = fma(-xr.y, y.y, v.x);
              v.y = fma(-xr.y, y.x, v.y); v.y = fma(xr.x, y.y, v.y);
            }
          }
          if (ti == jj + 1 && tk == jj + 1) {
            CT& v = a[mi][J0 * (J0 + 1) / 2 + J0];
            R d2 = v.x;
            if (!(d2 > (R)0)) { atomicOr(status, 1); d2 = (R)1; }
            const R inv = rsq(d2);
            v = mkc<CT>(d2 * inv, 0);
            sInv[mi * NPAD + j + 1] = inv;
          }
        }
      }
      __syncthreads();
    }
    if (J0 + 1 < NB) {
      // rank-16 update of the trailing blocks (I, J), J0 < J <= I (upper halves of diagonal blocks
      // are updated too and never read)
#pragma unroll
      for (int mi = 0; mi < MPC; ++mi) {
        const CT* pan = sPan + (size_t)mi * LA_BLK * NPAD;
        for (int k = 0; k < LA_BLK; ++k) {
          CT xr[NB], yc[NB];
#pragma unroll
          for (int I = J0 + 1; I < NB; ++I) {
            xr[I] = pan[k * NPAD + LA_BLK * I + ti];
            yc[I] = pan[k * NPAD + LA_BLK * I + tk];
          }
#pragma unroll
          for (int I = J0 + 1; I < NB; ++I)
#pragma unroll
            for (int J = J0 + 1; J <= I; ++J) {
              CT& v = a[mi][I * (I + 1) / 2 + J];
              v.x = fma(-xr[I].x, yc[J].x, v.x); v.x = fma(-xr[I].y, yc[J].y, v.x);
              v.y = fma(-xr[I].y, yc[J].x, v.y); v.y = fma(xr[I].x, yc[J].y, v.y);
            }
        }
      }
      if (tid == 0) {   // first pivot of the next panel
#pragma unroll
        for (int mi = 0; mi < MPC; ++mi) {
          CT& v = a[mi][(J0 + 1) * (J0 + 2) / 2 + J0 + 1];
          R d2 = v.x;
          if (!(d2 > (R)0)) { atomicOr(status, 1); d2 = (R)1; }
          const R inv = rsq(d2);
          v = mkc<CT>(d2 * inv, 0);
          sInv[mi * NPAD + LA_BLK * (J0 + 1)] = inv;
        }
      }
      __syncthreads();
    }
  }

#pragma unroll
  for (int mi = 0; mi < MPC; ++mi) {
    CT* F = factors + (size_t)bsv[mi] * L.fsize;
    const bool store = bsv[mi] < L.nsub;
#pragma unroll
    for (int I = 0; I < NB; ++I)
#pragma unroll
      for (int J = 0; J <= I; ++J) {
        if (I == J) {
          if (ti >= tk) sDiag[(mi * NB + I) * 256 + ti * LA_BLK + tk] = a[mi][I * (I + 1) / 2 + J];
        } else if (store) {
          F[(size_t)(I * (I + 1) / 2 + J) * 256 + ti * LA_BLK + tk] = a[mi][I * (I + 1) / 2 + J];
        }
      }
  }
  __syncthreads();
  if (tid < MPC * NB * LA_BLK) {
    const int mi = tid / (NB * LA_BLK), rem = tid - mi * NB * LA_BLK;
    const int I = rem / LA_BLK, jj = rem % LA_BLK, base = LA_BLK * I;
    int bm = 0;
#pragma unroll
    for (int u = 0; u < MPC; ++u) if (u == mi) bm = bsv[u];
    if (bm < L.nsub) {
      const CT* Ld = sDiag + (mi * NB + I) * 256;
      const R* Inv = sInv + mi * NPAD;
      CT x[LA_BLK];
#pragma unroll
      for (int i = 0; i < LA_BLK; ++i) {
        CT acc = mkc<CT>(0, 0);
#pragma unroll
        for (int k = 0; k < i; ++k)
          if (k >= jj) cfma(acc, Ld[i * LA_BLK + k], x[k]);
        const R rinv = Inv[base + i];
        if (i < jj) x[i] = mkc<CT>(0, 0);
        else if (i == jj) x[i] = mkc<CT>(rinv, 0);
        else x[i] = mkc<CT>(-acc.x * rinv, -acc.y * rinv);
      }
      CT* D = factors + (size_t)bm * L.fsize + (size_t)(I * (I + 1) / 2 + I) * 256;
#pragma unroll
      for (int i = 0; i < LA_BLK; ++i) D[i * LA_BLK + jj] = x[i];
    }
  }
}

// ======================================================================== wide subvolumes
// Finest-level subvolumes of up to 256 unknowns (4 x 4 x 4 points x K = 4 in 3D, 8 x 8 x 4 in 2D).
// Their factor (136 blocks: 557 KB complex128, 279 KB complex64) fits in no CTA's shared memory, so
// one 256-thread CTA per subvolume factorises left-looking by 16-column block columns directly in
// the factor store: block column J is assembled in registers, updated with the finished block
// columns 0..J-1 read back from global memory (recently written by the same CTA, so mostly L2
// hits), its diagonal block is factorised in shared memory, the blocks below it are divided by it,
// and the column is stored.  Entries of G_UU come from closed forms of H and H^2 on the grid, built
// once per subvolume into a shared-memory table of (H, H^2) over its point pairs.
constexpr int kWidePtsMax = 64;   // grid points of a wide subvolume
// row stride of the (H, H^2) pair table: odd, so that the rows of one column a warp reads spread over
// the banks
constexpr int kHHStride = kWidePtsMax + 1;

// Two consecutive complex entries (16-byte aligned), as one vector load where the type allows.
template <typename CT> struct CPair;
template <> struct CPair<float2> {
  float4 v;
  __device__ __forceinline__ void load(const float2* p) { v = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void load_zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ float2 a() const { return make_float2(v.x, v.y); }
  __device__ __forceinline__ float2 b() const { return make_float2(v.z, v.w); }
};
template <> struct CPair<double2> {
  double2 a_, b_;
  __device__ __forceinline__ void load(const double2* p) { a_ = __ldg(p); b_ = __ldg(p + 1); }
  __device__ __forceinline__ void load_zero() { a_ = make_double2(0.0, 0.0); b_ = a_; }
  __device__ __forceinline__ double2 a() const { return a_; }
  __device__ __forceinline__ double2 b() const { return b_; }
};
// the same pair from shared memory
__device__ __forceinline__ CPair<float2> lds_pair(const float2* p) {
  CPair<float2> r;
  r.v = *reinterpret_cast<const float4*>(p);
  return r;
}
__device__ __forceinline__ CPair<double2> lds_pair(const double2* p) {
  CPair<double2> r;
  r.a_ = p[0];
  r.b_ = p[1];
  return r;
}

// L2 eviction-priority policies and the loads that carry them.  The sweep reads each factor block
// twice, forward then backward; a launch's forward-read blocks outgrow L2 before the backward pass
// reaches them unless the single-use streams (the backward reads themselves, c and f) give way first.
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ unsigned long long l2_evict_last() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ float4 ldg_policy(const float4* p, unsigned long long pol) {
  float4 v;
  asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ float2 ldg_policy(const float2* p, unsigned long long pol) {
  float2 v;
  asm("ld.global.nc.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
  return v;
}
// coherent loads (the array is written by the same launch elsewhere) with a policy
__device__ __forceinline__ float2 ld_policy(const float2* p, unsigned long long pol) {
  float2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ double2 ld_policy(const double2* p, unsigned long long pol) {
  double2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(pol));
  return v;
}

// Asynchronous copy (cp.async) of one complex element global -> shared; cp_async_wait_all waits for the
// calling thread's copies.
__device__ __forceinline__ void cp_async_elem(float2* sdst, const float2* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)), "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async_elem(double2* sdst, const double2* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)), "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// the same with zero fill (nothing read) where valid is false
__device__ __forceinline__ void cp_async_elem_zf(float2* sdst, const float2* gsrc, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)),
               "l"(gsrc), "r"(valid ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_elem_zf(double2* sdst, const double2* gsrc, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)),
               "l"(gsrc), "r"(valid ? 16 : 0)
               : "memory");
}
// 16 bytes, both addresses 16-byte aligned
__device__ __forceinline__ void cp_async16_zf(void* sdst, const void* gsrc, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)),
               "l"(gsrc), "r"(valid ? 16 : 0)
               : "memory");
}
// one real value
__device__ __forceinline__ void cp_async_real(float* sdst, const float* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)), "l"(gsrc)
               : "memory");
}
__device__ __forceinline__ void cp_async_real(double* sdst, const double* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(sdst)), "l"(gsrc)
               : "memory");
}

// Shared-memory layout of the wide factorisation (bytes), for the padded size npad.
// Rows of the two shared-memory panels are padded so that the transposed stores of the block row and the
// column-wise accesses of the diagonal block spread over the banks: 17 entries for the block column,
// 18 for the block row (whose rows the update reads as 16-byte pairs, so they start 16-byte aligned).
constexpr int kWideStride = LA_BLK + 1;
constexpr int kRowStride = LA_BLK + 2;
__host__ __device__ constexpr size_t wide_factor_smem(int npad, size_t csize, size_t rsize) {
  return csize * ((size_t)(npad - LA_BLK) * kRowStride     // block row J+1, transposed (then the block (J+1, J))
                  + (size_t)npad * kWideStride             // the block column's rows at their absolute index
                  + 256)                                   // inv(L_JJ)^dagger, [k][c]
         + rsize * (LA_NPAIR * LA_KMAX * LA_KMAX + 3 * kWidePtsMax + LA_BLK) + sizeof(int) * kWidePtsMax
         + csize * (size_t)kWidePtsMax * kHHStride      // (H, H^2) of every point pair
         + rsize * 2 * LA_KMAX * LA_KMAX;               // P_HI - P_IH and P_XI - P_IX
}

// H_pq and (H^2)_pq of the finest-level operator H = -1/2 Laplacian + V0 for grid points p, q of one
// subvolume: D = dsum + V0 on the diagonal, -w_a = -1/(2 h_a^2) between neighbours along axis a,
// and H^2 by the paths of length two inside the grid (Dirichlet walls: the diagonal of H^2 counts
// only in-grid neighbours, nb2 = sum_a w_a^2 over them).
template <typename R>
__device__ __forceinline__ void wide_h_h2(int dx, int dy, int dz, R Dp, R Dq, R nb2p, R wx, R wy, R wz, R& H,
                                          R& H2) {
  const int ax = abs(dx), ay = abs(dy), az = abs(dz), a1 = ax + ay + az;
  H = 0;
  H2 = 0;
  if (a1 == 0) {
    H = Dp;
    H2 = Dp * Dp + nb2p;
  } else if (a1 == 1) {
    const R w = ax ? wx : (ay ? wy : wz);
    H = -w;
    H2 = -w * (Dp + Dq);
  } else if (a1 == 2) {
    if (ax == 2) H2 = wx * wx;
    else if (ay == 2) H2 = wy * wy;
    else if (az == 2) H2 = wz * wz;
    else H2 = 2 * (ax ? wx : wy) * (az ? wz : wy);
  }
}

// Shared-memory tables of the wide assembly: sHH[i * kHHStride + j] = (H_ij, (H^2)_ij) for the
// subvolume's points, sP the nine K x K products P_kk' = R_k^T Wt R_k' (Theta = phase x P) in the pair
// order (0,0) (0,1) (0,2) (1,0) (1,1) (1,2) (2,0) (2,1) (2,2) of (I, H, X), sPd = (P_01 - P_10, P_02 - P_20)
// (phases: (0,1), (0,2) +i; (1,0), (2,0) -i; the others real), sX the laser coordinate of each point.
template <typename R>
struct WideTables {
  typedef typename C2<R>::T CT;
  const CT* sHH;
  const R *sP, *sPd, *sX;
};
// The point and time function of one row of G_UU, decoded once per row.
template <typename R>
struct WideRow {
  int r, i, m;
  R xp;
};
template <typename R>
__device__ __forceinline__ WideRow<R> wide_row(int r, const FastDiv& dK, int K, const R* sX) {
  WideRow<R> w;
  w.r = r;
  w.i = fdiv(r, dK);
  w.m = r - w.i * K;
  w.xp = sX[w.i < kWidePtsMax ? w.i : 0];
  return w;
}

// Assembles G_UU[r, c] (r, c < npad; identity outside the n true unknowns).
template <typename R>
__device__ __forceinline__ typename C2<R>::T wide_entry(const WideRow<R>& w, int c, int n, const FastDiv& dK, int K,
                                                     const WideTables<R>& T) {
  typedef typename C2<R>::T CT;
  if (w.r >= n || c >= n) return mkc<CT>((R)(w.r == c ? 1 : 0), (R)0);
  const int j = fdiv(c, dK), nn = c - j * K;
  const CT hh = T.sHH[w.i * kHHStride + j];
  const R H = hh.x, H2 = hh.y;
  const int KK = K * K, mn = w.m * K + nn;
  const R xp = w.xp, xq = T.sX[j];
  R re = H2 * T.sP[4 * KK + mn] + H * (xq * T.sP[5 * KK + mn] + xp * T.sP[7 * KK + mn]);
  R im = H * T.sPd[mn];
  if (w.i == j) {
    re += T.sP[mn] + xp * xp * T.sP[8 * KK + mn];
    im += xp * T.sPd[KK + mn];
  }
  return mkc<CT>(re, im);
}

// Row r of block column Jc, columns c0 .. c0 + CPT - 1, assembled: acc[c] = G[r][16 Jc + c0 + c]
// (zero for a block beyond the band).  wide_partial_update then subtracts the finished block columns.
template <typename R, int CPT>
__device__ __forceinline__ void wide_assemble(int Jc, int band, int r, int c0, int n, const FastDiv& dK, int K,
                                              const WideTables<R>& T, typename C2<R>::T* acc) {
  typedef typename C2<R>::T CT;
  if ((r >> 4) - Jc > band) {
#pragma unroll
    for (int q = 0; q < CPT; ++q) acc[q] = mkc<CT>(0, 0);
    return;
  }
  const WideRow<R> w = wide_row<R>(r, dK, K, T.sX);
#pragma unroll
  for (int q = 0; q < CPT; ++q) acc[q] = wide_entry<R>(w, LA_BLK * Jc + c0 + q, n, dK, K, T);
}

// acc[c] -= sum_{k < 16 kb_end} L[r][k] conj(L[16 Jc + c0 + c][k]) over the finished block columns inside
// the band: row r's blocks read back from the factor store, block row Jc transposed in sRow.
template <typename R, int CPT>
__device__ __forceinline__ void wide_partial_update(int Jc, int kb_end, int band, int r, int c0,
                                                    const typename C2<R>::T* __restrict__ F,
                                                    const typename C2<R>::T* sRow, typename C2<R>::T* acc) {
  typedef typename C2<R>::T CT;
  const int I = r >> 4;
  if (I - Jc > band) return;   // a block beyond the band: zero, nothing to update
  // the blocks (I, Kb) with I - Kb > band are zero: the sum starts at Kb = I - band
  const int kb_begin = I - band > 0 ? I - band : 0;
  for (int h = 2 * kb_begin; h < 2 * kb_end; ++h) {   // half a finished block row (8 columns k) at a time
    const int Kb = h >> 1, k0 = (h & 1) * (LA_BLK / 2);
    const CT* src = F + (size_t)tri_index(I, Kb) * 256 + (r & 15) * LA_BLK + k0;
    CT v[LA_BLK / 2];
#pragma unroll
    for (int kk = 0; kk < LA_BLK / 2; ++kk) v[kk] = src[kk];
    const CT* rowk = sRow + ((size_t)Kb * LA_BLK + k0) * kRowStride + c0;
#pragma unroll
    for (int kk = 0; kk < LA_BLK / 2; ++kk) {
#pragma unroll
      for (int q = 0; q < CPT; q += (CPT > 1 ? 2 : 1)) {
        CT y[2];
        if (CPT > 1) {
          const CPair<CT> yp = lds_pair(rowk + kk * kRowStride + q);
          y[0] = yp.a();
          y[1] = yp.b();
        } else {
          y[0] = rowk[kk * kRowStride + q];
        }
#pragma unroll
        for (int u = 0; u < (CPT > 1 ? 2 : 1); ++u) {
          // acc -= v conj(y)
          acc[q + u].x = fma(-v[kk].x, y[u].x, acc[q + u].x); acc[q + u].x = fma(-v[kk].y, y[u].y, acc[q + u].x);
          acc[q + u].y = fma(-v[kk].y, y[u].x, acc[q + u].y); acc[q + u].y = fma(v[kk].x, y[u].y, acc[q + u].y);
        }
      }
    }
  }
}

// Shared state of the wide factorisation.
template <typename R>
struct WideSmem {
  typedef typename C2<R>::T CT;
  CT* sRow;   // [NPAD-16][18]: block row J' transposed, sRow[k][c] = L[16 J' + c][k]
  CT* sPan;   // [NPAD][17]: rows of the current block column at their absolute row index
  CT* sBT;    // [16][17]: sBT[k][c] = L[16 (J+1) + c][16 J + k] (the block (J+1, J)); in sRow's space
  CT* sInvT;  // [16][16]: sInvT[k][c] = conj(inv(L_JJ)[c][k])
  CT* sHH;    // [64][65]: (H, H^2) of the point pairs
  R *sP, *sPd, *sD, *sX, *sN, *sPiv;
  int* sXYZ;
  __device__ WideTables<R> tables() const { return WideTables<R>{sHH, sP, sPd, sX}; }
};

// Cholesky of the diagonal block of column J (rows 16 J .. 16 J + 15 of sPan) and its inverse in one
// sweep of 16 steps, by one warp.  Lane (i, h) = (lane % 16, lane / 16) updates row i's trailing entries of
// one column parity h and keeps the entries of parity h of row i of X = inv(L_JJ) in registers: X starts
// as the identity, and step j divides row j by L[j][j] and subtracts L[i][j] times it from the rows i > j
// (row j of X is final after step j), so the inverse costs no second chain of dependent steps.
template <typename R>
__device__ __forceinline__ void wide_diag(int J, const WideSmem<R>& S, typename C2<R>::T* F, int* status) {
  typedef typename C2<R>::T CT;
  const int lane = threadIdx.x & 31, ri = lane & 15, half = lane >> 4;
  CT* D = S.sPan + (size_t)LA_BLK * J * kWideStride;   // the diagonal block's rows
  CT x[LA_BLK / 2];                                     // X[ri][2 u + half]
#pragma unroll
  for (int u = 0; u < LA_BLK / 2; ++u) x[u] = mkc<CT>((R)(2 * u + half == ri ? 1 : 0), (R)0);
  for (int j = 0; j < LA_BLK; ++j) {
    R d2 = D[j * kWideStride + j].x;
    if (!(d2 > (R)0)) {
      if (lane == 0) atomicOr(status, 1);
      d2 = (R)1;
    }
    const R inv = rsq(d2);
    CT lij = mkc<CT>(0, 0);
    if (ri > j) {
      const CT v = D[ri * kWideStride + j];
      lij = mkc<CT>(v.x * inv, v.y * inv);
    }
    __syncwarp();
    if (ri > j && half == 0) D[ri * kWideStride + j] = lij;
    if (lane == j) D[j * kWideStride + j] = mkc<CT>(d2 * inv, (R)0);
    // X: row j /= L[j][j] (its lanes), then rows i > j -= L[i][j] X[j]; X[j][c] comes from lane (j, h)
#pragma unroll
    for (int u = 0; u < LA_BLK / 2; ++u) {
      if (ri == j) x[u] = mkc<CT>(x[u].x * inv, x[u].y * inv);
      CT xj;
      xj.x = __shfl_sync(0xffffffffu, x[u].x, j + 16 * half);
      xj.y = __shfl_sync(0xffffffffu, x[u].y, j + 16 * half);
      if (ri > j) {   // x -= L[i][j] X[j]
        x[u].x -= lij.x * xj.x - lij.y * xj.y;
        x[u].y -= lij.x * xj.y + lij.y * xj.x;
      }
    }
    __syncwarp();
    // trailing entries (i, k), j < k <= i: A[i][k] -= L[i][j] conj(L[k][j])
    if (ri > j) {
      for (int k = j + 1 + half; k <= ri; k += 2) {
        const CT lk = D[k * kWideStride + j];
        CT v = D[ri * kWideStride + k];
        v.x -= lij.x * lk.x + lij.y * lk.y;
        v.y -= lij.y * lk.x - lij.x * lk.y;
        D[ri * kWideStride + k] = v;
      }
    }
    __syncwarp();
  }
  // the inverse as the stored diagonal block (row ri, columns 2 u + half), and sInvT[k][c] = conj(X[c][k])
#pragma unroll
  for (int u = 0; u < LA_BLK / 2; ++u) {
    const int c = 2 * u + half;
    if (lane < 32) {
      F[(size_t)tri_index(J, J) * 256 + ri * LA_BLK + c] = x[u];
      S.sInvT[c * LA_BLK + ri] = mkc<CT>(x[u].x, -x[u].y);
    }
  }
}

// Named barrier of warps 1..7 (the lookahead update's threads).
__device__ __forceinline__ void wide_bar() { asm volatile("bar.sync 1, 224;" ::: "memory"); }

// One block column J with lookahead: warp 0 factorises J's diagonal block while warps 1..7 assemble block
// column J+1 and update it with the finished block columns 0..J-1; then all threads divide J's rows below
// by L_JJ, and warps 1..7 add block column J's contribution to J+1 from shared memory.
template <typename R, int NPAD, int CPT>
__device__ __forceinline__ void wide_column_step(int J, int band, int n, const FastDiv& dK, int K,
                                                 typename C2<R>::T* F, const WideSmem<R>& S, int* status) {
  typedef typename C2<R>::T CT;
  constexpr int NB = NPAD / LA_BLK;
  constexpr int TPR = LA_BLK / CPT;
  const int tid = threadIdx.x;
  const bool next = J + 1 < NB;
  const int RJ1 = NPAD - LA_BLK * (J + 1);            // rows of block column J+1
  // warps 1..7 own rows q' = t' / TPR of block column J+1 (t' = tid - 32); rows beyond 224 / TPR
  // (block column 1 of a 256-unknown matrix has 240) fall to warp 0 after its diagonal work
  const int tl = tid - 32;
  const int q_own = tid >= 32 ? tl / TPR : 224 / TPR + (tid & 31);
  const int c0 = tid >= 32 ? (tl % TPR) * CPT : 0;
  const bool own = next && q_own < RJ1 && (tid >= 32 || (TPR == 1 && (tid & 31) < LA_BLK));
  const int r_own = LA_BLK * (J + 1) + q_own;
  CT acc[CPT];
  if (tid < 32) {
    wide_diag<R>(J, S, F, status);
  } else if (next) {
    // block row J+1's finished blocks (J+1, Kb < J) inside the band, transposed, every copy in flight at once
    const int kb0 = J + 1 - band > 0 ? J + 1 - band : 0;
    for (int t = kb0 * 256 + tl; t < J * 256; t += 224) {
      const int Kb = t >> 8, w = t & 255, c = w >> 4, kk = w & 15;
      cp_async_elem(S.sRow + (Kb * LA_BLK + kk) * kRowStride + c, F + (size_t)tri_index(J + 1, Kb) * 256 + w);
    }
    // the entries of G are assembled while the copies are in flight
    if (own) wide_assemble<R, CPT>(J + 1, band, r_own, c0, n, dK, K, S.tables(), acc);
    cp_async_wait_all();
    wide_bar();
    if (own) wide_partial_update<R, CPT>(J + 1, J, band, r_own, c0, F, S.sRow, acc);
  }
  __syncthreads();
  if (tid < 32 && own)   // warp 0's rows of block column 1 (no finished column before it)
    wide_assemble<R, CPT>(J + 1, band, r_own, c0, n, dK, K, S.tables(), acc);
  // rows below the diagonal block, one row per thread: L[r][c] = sum_{k <= c} A[r][k] conj(inv(L_JJ)[c][k])
  // (the row's entries in registers, sInvT's rows read as 16-byte pairs), written to the factor store and
  // back to the row in place; the rows of the block (J+1, J) also go to sBT for the update below
  // (rows beyond the band hold exact zeros, which stay zeros)
  for (int q = tid; q < RJ1 && q < LA_BLK * band; q += kFactorThreads) {
    const int rr = LA_BLK * (J + 1) + q;
    CT* row = S.sPan + (size_t)rr * kWideStride;
    CT a[LA_BLK], l[LA_BLK];
#pragma unroll
    for (int k = 0; k < LA_BLK; ++k) {
      a[k] = row[k];
      l[k] = mkc<CT>(0, 0);
    }
#pragma unroll
    for (int k = 0; k < LA_BLK; ++k) {
#pragma unroll
      for (int c = k - (k & 1); c < LA_BLK; c += 2) {   // inv is lower triangular: only c >= k contribute
        const CPair<CT> ip = lds_pair(S.sInvT + k * LA_BLK + c);
        cfma(l[c], a[k], ip.a());
        cfma(l[c + 1], a[k], ip.b());
      }
    }
#pragma unroll
    for (int c = 0; c < LA_BLK; ++c) row[c] = l[c];
    if ((rr >> 4) == J + 1) {
#pragma unroll
      for (int c = 0; c < LA_BLK; ++c) S.sBT[c * kWideStride + (rr & 15)] = l[c];
    }
  }
  __syncthreads();
  // the divided rows to the factor store, consecutive threads on consecutive entries
  for (int e = tid; e < RJ1 * LA_BLK; e += kFactorThreads) {
    const int rr = LA_BLK * (J + 1) + (e >> 4), c = e & 15;
    F[(size_t)tri_index(rr >> 4, J) * 256 + (rr & 15) * LA_BLK + c] = S.sPan[(size_t)rr * kWideStride + c];
  }
  __syncthreads();   // the rows are overwritten below with block column J+1
  if (own && (r_own >> 4) - J <= band) {
    // block column J's contribution: acc[c] -= sum_k L[r][16 J + k] conj(L[16 (J+1) + c][16 J + k])
    // (zero for rows whose block (I, J) is beyond the band)
    const CT* a = S.sPan + (size_t)r_own * kWideStride;
#pragma unroll
    for (int k = 0; k < LA_BLK; ++k) {
      const CT lr = a[k];
#pragma unroll
      for (int q = 0; q < CPT; ++q) {
        const CT y = S.sBT[k * kWideStride + c0 + q];
        acc[q].x = fma(-lr.x, y.x, acc[q].x); acc[q].x = fma(-lr.y, y.y, acc[q].x);
        acc[q].y = fma(-lr.y, y.x, acc[q].y); acc[q].y = fma(lr.x, y.y, acc[q].y);
      }
    }
  }
  __syncwarp();
  if (own) {
#pragma unroll
    for (int q = 0; q < CPT; ++q) S.sPan[(size_t)r_own * kWideStride + c0 + q] = acc[q];
  }
  __syncthreads();
}

// Fills the shared-memory tables of the wide assembly for the subvolume with origin o and extent e; all
// threads of the CTA, synchronised on return.
template <typename R>
__device__ __forceinline__ void wide_tables(const LevelGeom& L, const FineOp& g, const TimeMats* __restrict__ tm,
                                            const int o[3], const int e[3], R* sP, R* sPd, R* sD, R* sX, R* sN,
                                            int* sXYZ, typename C2<R>::T* sHH) {
  typedef typename C2<R>::T CT;
  const int tid = threadIdx.x, nthr = blockDim.x, K = tm->K, KK = K * K, npts = e[0] * e[1] * e[2];
  for (int i = tid; i < LA_NPAIR * KK; i += nthr) sP[i] = (R)tm->P[i / KK][i % KK];
  const R wx = (R)(0.5 * g.ih2[0]), wy = (R)(0.5 * g.ih2[1]), wz = (R)(0.5 * g.ih2[2]);
  for (int i = tid; i < npts; i += nthr) {
    int lx, ly, lz;
    local_coords(i, e, lx, ly, lz);
    const int px = o[0] + lx, py = o[1] + ly, pz = o[2] + lz;
    sD[i] = (R)(g.dsum + g.V0[(pz * g.n[1] + py) * g.n[0] + px]);
    sX[i] = (R)fine_x(g, px, py, pz);
    // unused axes have n = 1 and w = 0
    const int cx = (px > 0 ? 1 : 0) + (px + 1 < g.n[0] ? 1 : 0), cy = (py > 0 ? 1 : 0) + (py + 1 < g.n[1] ? 1 : 0),
              cz = (pz > 0 ? 1 : 0) + (pz + 1 < g.n[2] ? 1 : 0);
    sN[i] = wx * wx * (R)cx + wy * wy * (R)cy + wz * wz * (R)cz;
    sXYZ[i] = lx | (ly << 8) | (lz << 16);
  }
  __syncthreads();
  for (int p = tid; p < npts * npts; p += nthr) {
    const int i = p / npts, j = p - i * npts;
    const int pi = sXYZ[i], pj = sXYZ[j];
    const int dx = (pj & 255) - (pi & 255), dy = ((pj >> 8) & 255) - ((pi >> 8) & 255), dz = (pj >> 16) - (pi >> 16);
    R H, H2;
    wide_h_h2<R>(dx, dy, dz, sD[i], sD[j], sN[i], wx, wy, wz, H, H2);
    sHH[i * kHHStride + j] = mkc<CT>(H, H2);
  }
  for (int i = tid; i < KK; i += nthr) {
    sPd[i] = sP[1 * KK + i] - sP[3 * KK + i];
    sPd[KK + i] = sP[2 * KK + i] - sP[6 * KK + i];
  }
  __syncthreads();
}

template <typename R, int NPAD>
__global__ void __launch_bounds__(kFactorThreads, sizeof(R) == 4 ? 2 : 1)
k_factor_wide(LevelGeom L, FineOp g, const TimeMats* __restrict__ tm, typename C2<R>::T* __restrict__ factors,
              int* __restrict__ status) {
  typedef typename C2<R>::T CT;
  constexpr int NB = NPAD / LA_BLK;
  extern __shared__ __align__(16) unsigned char smem[];
  WideSmem<R> S;
  S.sRow = reinterpret_cast<CT*>(smem);
  S.sBT = S.sRow;   // written after the lookahead update has read sRow, read before sRow is refilled
  S.sPan = S.sRow + (size_t)(NPAD - LA_BLK) * kRowStride;
  S.sInvT = S.sPan + (size_t)NPAD * kWideStride;
  S.sP = reinterpret_cast<R*>(S.sInvT + 256);
  S.sD = S.sP + LA_NPAIR * LA_KMAX * LA_KMAX;
  S.sX = S.sD + kWidePtsMax;
  S.sN = S.sX + kWidePtsMax;
  S.sPiv = S.sN + kWidePtsMax;
  S.sXYZ = reinterpret_cast<int*>(S.sPiv + LA_BLK);
  S.sHH = reinterpret_cast<CT*>(S.sXYZ + kWidePtsMax);
  S.sPd = reinterpret_cast<R*>(S.sHH + kWidePtsMax * kHHStride);

  const int tid = threadIdx.x;
  const int K = tm->K, KK = K * K;
  const int b = blockIdx.x;
  int o[3], e[3];
  subvol_box(L, b, o, e);
  const int npts = e[0] * e[1] * e[2], n = npts * K;
  CT* F = factors + (size_t)b * L.fsize;
  wide_tables<R>(L, g, tm, o, e, S.sP, S.sPd, S.sD, S.sX, S.sN, S.sXYZ, S.sHH);
  const FastDiv dK = L.fd_K;
  const WideTables<R> T = S.tables();
  // block column 0: assembled only, one row per thread
  if (tid < NPAD) {
    CT a0[LA_BLK];
    const WideRow<R> w = wide_row<R>(tid, dK, K, S.sX);
#pragma unroll
    for (int q = 0; q < LA_BLK; ++q) a0[q] = wide_entry<R>(w, q, n, dK, K, T);
#pragma unroll
    for (int q = 0; q < LA_BLK; ++q) S.sPan[(size_t)tid * kWideStride + q] = a0[q];
  }
  __syncthreads();
  for (int J = 0; J < NB; ++J) {
    // threads per row of block column J+1 over the 224 lookahead threads
    const int RJ1 = NPAD - LA_BLK * (J + 1);
    int tpr = 1;
    while (tpr < 8 && 2 * tpr * RJ1 <= 224) tpr *= 2;
    switch (tpr) {
      case 1: wide_column_step<R, NPAD, 16>(J, L.band, n, dK, K, F, S, status); break;
      case 2: wide_column_step<R, NPAD, 8>(J, L.band, n, dK, K, F, S, status); break;
      case 4: wide_column_step<R, NPAD, 4>(J, L.band, n, dK, K, F, S, status); break;
      default: wide_column_step<R, NPAD, 2>(J, L.band, n, dK, K, F, S, status); break;
    }
  }
}

// ------------------------------------------------------------------------ banded, window in registers
// Wide complex64 factors whose block band is at most W: blocked right-looking Cholesky with the active
// window in registers.  While block column J is eliminated, the trailing blocks (J + i, J + j),
// 1 <= j <= i <= W, are the only ones that change (no fill outside the envelope), so thread (ti, tk) keeps
// its entry (ti, tk) of each of them in registers and the window moves one block along the diagonal per
// column; a new block row is assembled as it enters.  Per column, three barriers:
//   panel   L_i = A_i inv(L_JJ)^dagger for the W blocks below the diagonal, to the factor store and,
//           k-major, to shared memory;
//   column  the blocks (i, 1) take the rank-16 update first and go to shared memory as the next column;
//   rest    a ninth warp factorises and inverts the next diagonal block (lookahead) while the others apply
//           the rank-16 update to the remaining blocks and assemble the row that enters.
// The factor is written once and never read back.
// Its diagonal superblocks of kSuper block rows hold the inverse of L's superblock instead of L, so that the
// triangular solves take NB / 4 steps of larger mat-vecs instead of NB (factor_is_super).  The inverse X is
// built along with the elimination: the blocks Z_IC = sum_{C <= k < I} L_Ik X_kC grow by one term per column,
// and X_IC = -inv(L_II) Z_IC when the diagonal block I is inverted; 16 block products per superblock, 11%
// more multiplications.
// 96^3, K = 4, 4x4x4 subvolumes (13,824 factors of 256 unknowns, W = 8): 8.24 ms = 21 TFLOP/s of banded flops,
// bound by instruction issue (6.88 ms without the superblocks' inverses, 67% of the issue slots and 46% of
// the FMA pipe busy); 11.1 ms with the left-looking
// factorisation below, which waits on its own earlier blocks in L2 and on a diagonal step three times
// as long.  A diagonal step by one of the eight warps instead of a ninth: 9.6 ms.
constexpr int kSuper = 4;
template <int W> struct BandSmem {
  // the panel and the inverse hold two columns k, k + 1 of a row next to each other, one 16-byte load for
  // both; rows of a panel pair: one more than the window, so that the transposed stores spread over the banks
  static constexpr int kPanStride = 2 * (LA_BLK * W + 1);
  // complex entries: column blocks, inverse, two row buffers of the diagonal step, panel, the blocks (i, 1),
  // the inverse's own layout of two columns, the superblock's inverse
  static constexpr int kComplex =
      (W + 1) * LA_BLK * kRowStride + 256 + 32 + LA_BLK / 2 * kPanStride + 256 * W + 512 + 6 * 256;
};
template <typename R, int W>
__host__ __device__ constexpr size_t band_factor_smem() {
  return 2 * sizeof(R) * ((size_t)BandSmem<W>::kComplex + (size_t)kWidePtsMax * kHHStride) +
         sizeof(R) * (LA_NPAIR * LA_KMAX * LA_KMAX + 3 * kWidePtsMax + 2 * LA_KMAX * LA_KMAX) +
         sizeof(int) * kWidePtsMax;
}

// Cholesky factor and inverse of the 16 x 16 block D (row stride kRowStride) by one warp, in place: step j
// scales column j to L and frees it, and the inverse X of L fills the freed columns, so lane (r, h) =
// (lane % 16, lane / 16) holds one value per column of parity h of row r, A[r][c] for c > j and X[r][c] for
// c <= j, and every step updates the rows r > j by v[c] -= L_rj w[c] with the row w[c] = conj(L_cj) for
// c > j, X[j][c] for c <= j (passed through shared memory, read as 16-byte pairs).  Ends with X = inv(L).
template <typename CT>
__device__ __forceinline__ void band_diag(const CT* D, CT* sInvT, CT* sX, CT* buf, CT* Fdiag, int* status) {
  typedef typename Re<CT>::T R;
  const int lane = threadIdx.x & 31, r = lane & 15, h = lane >> 4;
  CT v[LA_BLK / 2];   // column 2 u + h
#pragma unroll
  for (int u = 0; u < LA_BLK / 2; ++u) v[u] = D[r * kRowStride + 2 * u + h];
#pragma unroll
  for (int j = 0; j < LA_BLK; ++j) {
    const int uj = j >> 1, hj = j & 1;
    CT l;
    l.x = __shfl_sync(0xffffffffu, v[uj].x, r + 16 * hj);
    l.y = __shfl_sync(0xffffffffu, v[uj].y, r + 16 * hj);
    R d2 = __shfl_sync(0xffffffffu, v[uj].x, j + 16 * hj);
    if (!(d2 > (R)0)) {
      if (lane == 0) atomicOr(status, 1);
      d2 = (R)1;
    }
    const R inv = rsq(d2);
    l = r > j ? mkc<CT>(l.x * inv, l.y * inv) : mkc<CT>((R)0, (R)0);
    if (h == hj) v[uj] = mkc<CT>((R)(r == j ? 1 : 0), (R)0);   // column j now belongs to X
    CT* b = buf + (j & 1) * 16;   // [parity][8] columns
    if (r > j && h == 0) b[(r & 1) * 8 + (r >> 1)] = mkc<CT>(l.x, -l.y);
    if (r == j) {
#pragma unroll
      for (int u = 0; 2 * u <= j; ++u) {
        if (2 * u + h > j) continue;
        v[u] = mkc<CT>(v[u].x * inv, v[u].y * inv);
        b[h * 8 + u] = v[u];
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < LA_BLK / 2; u += 2) {
      const CPair<CT> p = lds_pair(b + h * 8 + u);
      const CT w0 = p.a(), w1 = p.b();
      CT &t0 = v[u], &t1 = v[u + 1];
      t0.x = fma(-l.x, w0.x, t0.x); t0.x = fma(l.y, w0.y, t0.x);
      t0.y = fma(-l.x, w0.y, t0.y); t0.y = fma(-l.y, w0.x, t0.y);
      t1.x = fma(-l.x, w1.x, t1.x); t1.x = fma(l.y, w1.y, t1.x);
      t1.y = fma(-l.x, w1.y, t1.y); t1.y = fma(-l.y, w1.x, t1.y);
    }
  }
#pragma unroll
  for (int u = 0; u < LA_BLK / 2; ++u) {
    const int c = 2 * u + h;
    if (c > r) v[u] = mkc<CT>((R)0, (R)0);
    Fdiag[r * LA_BLK + c] = v[u];
    sInvT[(c >> 1) * 32 + 2 * r + (c & 1)] = mkc<CT>(v[u].x, -v[u].y);
    sX[(r >> 1) * 32 + 2 * c + (r & 1)] = v[u];
  }
}

// v -= x conj(y)
template <typename CT>
__device__ __forceinline__ void band_fma(CT& v, const CT x, const CT y) {
  v.x = fma(-x.x, y.x, v.x); v.x = fma(-x.y, y.y, v.x);
  v.y = fma(-x.y, y.x, v.y); v.y = fma(x.x, y.y, v.y);
}
// Rank-16 update of the window blocks (i, j), I0 <= i <= I1, 2 <= j <= i: a(i, j) -= L_i L_j^dagger.
// a(i, j) is at (i - 2) (i - 1) / 2 + j - 2.
template <typename CT, int W, int I0, int I1>
__device__ __forceinline__ void band_update(CT (&a)[W * (W - 1) / 2], const CT* pan, int ti, int tk) {
#pragma unroll 1
  for (int k2 = 0; k2 < LA_BLK / 2; ++k2) {
    const CT* p = pan + k2 * BandSmem<W>::kPanStride;
    CPair<CT> x[I1 - I0 + 1];
#pragma unroll
    for (int i = I0; i <= I1; ++i) x[i - I0] = lds_pair(p + 2 * (LA_BLK * (i - 1) + ti));
#pragma unroll
    for (int j = 2; j <= I1; ++j) {
      const CPair<CT> y = lds_pair(p + 2 * (LA_BLK * (j - 1) + tk));
#pragma unroll
      for (int i = I0; i <= I1; ++i)
        if (j <= i) {
          CT& v = a[(i - 2) * (i - 1) / 2 + j - 2];
          band_fma(v, x[i - I0].a(), y.a());
          band_fma(v, x[i - I0].b(), y.b());
        }
    }
  }
}

static_assert(kSuper == 4, "the superblock inverse is written for four block rows");
// x[c] = X_Pc = -inv(L_PP) Z_Pc, c < P: rows ti of inv(L_PP) end at column ti, so warp ti / 2 stops there.
template <typename CT, int P>
__device__ __forceinline__ void band_inv_row(CT (&x)[kSuper - 1], const CT* sInvT, const CT* sZ, int ti, int tk) {
  CT v[P];
#pragma unroll
  for (int c = 0; c < P; ++c) v[c] = mkc<CT>(0, 0);
#pragma unroll 2
  for (int k2 = 0; k2 <= (ti >> 1); ++k2) {
    const CPair<CT> a = lds_pair(sInvT + k2 * 32 + 2 * ti);
#pragma unroll
    for (int c = 0; c < P; ++c) {
      const CPair<CT> z = lds_pair(sZ + (P * (P - 1) / 2 + c) * 256 + k2 * 32 + 2 * tk);
      cfma_conj(v[c], a.a(), z.a());
      cfma_conj(v[c], a.b(), z.b());
    }
  }
#pragma unroll
  for (int c = 0; c < P; ++c) x[c] = mkc<CT>(-v[c].x, -v[c].y);
}
// Z_ic += L_iP X_Pc for the superblock's rows i > P and columns c <= P (X_PP in xd).
template <typename CT, int W, int P>
__device__ __forceinline__ void band_inv_update(CT* sZ, const CT* xd, const CT* pan, int ti, int tk, int own) {
  CT z[kSuper - 1 - P][P + 1];
#pragma unroll
  for (int i = P + 1; i < kSuper; ++i)
#pragma unroll
    for (int c = 0; c <= P; ++c) z[i - P - 1][c] = c < P ? sZ[(i * (i - 1) / 2 + c) * 256 + own] : mkc<CT>(0, 0);
#pragma unroll 2
  for (int k2 = 0; k2 < LA_BLK / 2; ++k2) {
    CPair<CT> x[kSuper - 1 - P];
#pragma unroll
    for (int i = P + 1; i < kSuper; ++i)
      x[i - P - 1] = lds_pair(pan + k2 * BandSmem<W>::kPanStride + 2 * (LA_BLK * (i - P - 1) + ti));
#pragma unroll
    for (int c = 0; c <= P; ++c) {
      const CPair<CT> y = lds_pair((c < P ? sZ + (P * (P - 1) / 2 + c) * 256 : xd) + k2 * 32 + 2 * tk);
#pragma unroll
      for (int i = P + 1; i < kSuper; ++i) {
        cfma(z[i - P - 1][c], x[i - P - 1].a(), y.a());
        cfma(z[i - P - 1][c], x[i - P - 1].b(), y.b());
      }
    }
  }
#pragma unroll
  for (int i = P + 1; i < kSuper; ++i)
#pragma unroll
    for (int c = 0; c <= P; ++c) sZ[(i * (i - 1) / 2 + c) * 256 + own] = z[i - P - 1][c];
}

constexpr int kBandThreads = kFactorThreads + 32;
__device__ __forceinline__ void band_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

template <typename R, int NPAD, int W>
__global__ void __launch_bounds__(kBandThreads, 2)
k_factor_band(LevelGeom L, FineOp g, const TimeMats* __restrict__ tm, typename C2<R>::T* __restrict__ factors,
              int* __restrict__ status) {
  typedef typename C2<R>::T CT;
  static_assert(W % 4 == 0, "window rows are updated in groups of four");
  constexpr int NB = NPAD / LA_BLK, S = BandSmem<W>::kPanStride;
  extern __shared__ __align__(16) unsigned char smem[];
  CT* sA = reinterpret_cast<CT*>(smem);              // [(W + 1) * 16][18] the column's blocks, diagonal first
  CT* sInvT = sA + (W + 1) * LA_BLK * kRowStride;   // inv(L_JJ)^dagger, [k / 2][c][k % 2]
  CT* sBuf = sInvT + 256;                            // [2][16] rows of the diagonal step
  CT* sPan = sBuf + 32;                              // [8][S] the panel, [k / 2][row][k % 2]
  CT* sB = sPan + LA_BLK / 2 * S;                        // [W][256] the blocks (i, 1), each thread its own entries
  CT* sXd = sB + 256 * W;                            // [2][256] inv(L_JJ) of columns J and J + 1, [k / 2][c][k % 2]
  CT* sZ = sXd + 512;                                // [6][256] Z, then X, of the blocks (i, c) of the superblock
  CT* sHH = sZ + 6 * 256;                            // [64][65] (H, H^2) of the point pairs
  R* sP = reinterpret_cast<R*>(sHH + kWidePtsMax * kHHStride);
  R* sPd = sP + LA_NPAIR * LA_KMAX * LA_KMAX;
  R* sD = sPd + 2 * LA_KMAX * LA_KMAX;
  R* sX = sD + kWidePtsMax;
  R* sN = sX + kWidePtsMax;
  int* sXYZ = reinterpret_cast<int*>(sN + kWidePtsMax);

  const int tid = threadIdx.x, ti = tid >> 4, tk = tid & 15;
  const int K = tm->K, KK = K * K, band = L.band;
  int o[3], e[3];
  subvol_box(L, blockIdx.x, o, e);
  const int npts = e[0] * e[1] * e[2], n = npts * K;
  CT* F = factors + (size_t)blockIdx.x * L.fsize;
  wide_tables<R>(L, g, tm, o, e, sP, sPd, sD, sX, sN, sXYZ, sHH);
  const FastDiv dK = L.fd_K;
  const WideTables<R> T{sHH, sP, sPd, sX};
  // entry (ti, tk) of block (I, J) of G_UU; where K divides 16 its time functions do not depend on the block
  const bool kdiv = (LA_BLK % K) == 0;
  const int ppb = LA_BLK / K, pr = fdiv(ti, dK), pc = fdiv(tk, dK), mn = (ti - pr * K) * K + (tk - pc * K);
  auto entry = [&](int I, int J) {
    if (!kdiv) return wide_entry<R>(wide_row<R>(LA_BLK * I + ti, dK, K, sX), LA_BLK * J + tk, n, dK, K, T);
    const int i = I * ppb + pr, j = J * ppb + pc;
    if (i >= npts || j >= npts) return mkc<CT>((R)(I == J && ti == tk ? 1 : 0), (R)0);
    const CT hh = sHH[i * kHHStride + j];
    const R xp = sX[i], xq = sX[j];
    R re = hh.y * sP[4 * KK + mn] + hh.x * (xq * sP[5 * KK + mn] + xp * sP[7 * KK + mn]);
    R im = hh.x * sPd[mn];
    if (i == j) {
      re += sP[mn] + xp * xp * sP[8 * KK + mn];
      im += xp * sPd[KK + mn];
    }
    return mkc<CT>(re, im);
  };
  if (tid >= kFactorThreads) {   // the diagonal warp
    for (int J = 0; J < NB; ++J) {
      __syncthreads();   // column J is in sA
      band_diag<CT>(sA, sInvT, sXd + (J & 1) * 256, sBuf, F + (size_t)tri_index(J, J) * 256, status);
      __syncthreads();
    }
    return;
  }
#pragma unroll 1
  for (int i = 0; i <= W && i < NB; ++i) sA[(LA_BLK * i + ti) * kRowStride + tk] = entry(i, 0);
  __syncthreads();
#pragma unroll 1
  for (int i = 1; i <= W && i < NB; ++i) sB[(i - 1) * 256 + tid] = entry(i, 1);
  CT a[W * (W - 1) / 2];   // a(i, j) = block (J + i, J + j), 2 <= j <= i
#pragma unroll
  for (int i = 2; i <= W; ++i)
#pragma unroll
    for (int j = 2; j <= i; ++j) a[(i - 2) * (i - 1) / 2 + j - 2] = entry(i, j);
  __syncthreads();
#pragma unroll 1
  for (int J = 0; J < NB; ++J) {
    const int we = NB - 1 - J < W ? NB - 1 - J : W;   // blocks below the diagonal
    const int p = J % kSuper;                         // row J's place in its superblock
    // row J of the superblock's inverse: X_Jc = -inv(L_JJ) Z_Jc
    CT xr[kSuper - 1];
    if (p == 1) band_inv_row<CT, 1>(xr, sInvT, sZ, ti, tk);
    else if (p == 2) band_inv_row<CT, 2>(xr, sInvT, sZ, ti, tk);
    else if (p == 3) band_inv_row<CT, 3>(xr, sInvT, sZ, ti, tk);
#pragma unroll
    for (int c = 0; c < kSuper - 1; ++c)
      if (c < p) F[(size_t)tri_index(J, J - p + c) * 256 + tid] = xr[c];
    // panel, four blocks at a time
#pragma unroll 1
    for (int i0 = 1; i0 <= we; i0 += 4) {
      CT l[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) l[u] = mkc<CT>(0, 0);
      const CT* ar = sA + (LA_BLK * i0 + ti) * kRowStride;
#pragma unroll 2
      for (int k = 0; k < LA_BLK; k += 2) {
        const CPair<CT> iv = lds_pair(sInvT + k * LA_BLK + 2 * tk);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const CPair<CT> ap = lds_pair(ar + u * LA_BLK * kRowStride + k);
          cfma(l[u], ap.a(), iv.a());
          cfma(l[u], ap.b(), iv.b());
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u;
        if (i > we) break;
        sPan[(tk >> 1) * S + 2 * (LA_BLK * (i - 1) + ti) + (tk & 1)] = l[u];
        if (i <= band && i + p >= kSuper) F[(size_t)tri_index(J + i, J) * 256 + tid] = l[u];
      }
    }
    if (we == 0) break;
    band_bar();
    const int own = (ti >> 1) * 32 + 2 * tk + (ti & 1);   // this thread's entry of a [k / 2][c][k % 2] block
#pragma unroll
    for (int c = 0; c < kSuper - 1; ++c)
      if (c < p) sZ[(p * (p - 1) / 2 + c) * 256 + own] = xr[c];
    // next column: the blocks (i, 1), updated first, and the block that enters the band
#pragma unroll 1
    for (int i0 = 1; i0 <= we; i0 += 4) {
      CT v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = sB[(i0 - 1 + u) * 256 + tid];
#pragma unroll 2
      for (int k2 = 0; k2 < LA_BLK / 2; ++k2) {
        const CT* p = sPan + k2 * S;
        const CPair<CT> y = lds_pair(p + 2 * tk);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const CPair<CT> x = lds_pair(p + 2 * (LA_BLK * (i0 - 1 + u) + ti));
          band_fma(v[u], x.a(), y.a());
          band_fma(v[u], x.b(), y.b());
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) sA[(LA_BLK * (i0 - 1 + u) + ti) * kRowStride + tk] = v[u];
    }
    if (J + 1 + W < NB) sA[(LA_BLK * W + ti) * kRowStride + tk] = entry(J + 1 + W, J + 1);
    __syncthreads();
    if (p == 0) band_inv_update<CT, W, 0>(sZ, sXd + (J & 1) * 256, sPan, ti, tk, own);
    else if (p == 1) band_inv_update<CT, W, 1>(sZ, sXd + (J & 1) * 256, sPan, ti, tk, own);
    else if (p == 2) band_inv_update<CT, W, 2>(sZ, sXd + (J & 1) * 256, sPan, ti, tk, own);
    if (we > 1) {
      band_update<CT, W, 2, 4>(a, sPan, ti, tk);
      if constexpr (W > 4) {
        if (we > 6) band_update<CT, W, 5, W>(a, sPan, ti, tk);
        else if (we > 4) band_update<CT, W, 5, 6>(a, sPan, ti, tk);
      }
    }
    // move the window one block along the diagonal
#pragma unroll
    for (int i = 2; i <= W; ++i) sB[(i - 2) * 256 + tid] = a[(i - 2) * (i - 1) / 2];
#pragma unroll
    for (int i = 2; i < W; ++i)
#pragma unroll
      for (int j = 2; j <= i; ++j) a[(i - 2) * (i - 1) / 2 + j - 2] = a[(i - 1) * i / 2 + j - 1];
    if (J + 1 + W < NB) {
      sB[(W - 1) * 256 + tid] = entry(J + 1 + W, J + 2);
#pragma unroll
      for (int j = 2; j <= W; ++j) a[(W - 2) * (W - 1) / 2 + j - 2] = entry(J + 1 + W, J + 1 + j);
    }
    __syncthreads();
  }
}

// ======================================================================== triangular solves
// x = (L L^dagger)^{-1} rhs with the blocked factor F; rhs is overwritten by x.  Two warps (64
// threads, 4 lanes per row) do the block mat-vecs and synchronise with a named barrier; the other
// warps of the CTA skip the solve.  Four lanes per row keep the cross-lane reduction at two shuffle
// levels, which matters because every FP64 add issues on the slow FP64 pipe.  The caller
// synchronises the whole CTA before and after.
__device__ __forceinline__ void solve_bar() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

template <typename CT>
__device__ __forceinline__ CT reduce4(CT v) {
  v.x += __shfl_xor_sync(0xffffffffu, v.x, 1); v.y += __shfl_xor_sync(0xffffffffu, v.y, 1);
  v.x += __shfl_xor_sync(0xffffffffu, v.x, 2); v.y += __shfl_xor_sync(0xffffffffu, v.y, 2);
  return v;
}

template <typename CT, int NPAD, bool ENV>
__device__ __forceinline__ void subvol_solve_t(const LevelGeom& L, const CT* __restrict__ F, CT* rhs, CT* y, CT* tvec) {
  constexpr int NB = NPAD / LA_BLK;
  const int tid = threadIdx.x;
  if (tid >= 64) return;
  const int r = tid >> 2, l = tid & 3, r0 = r & 8;   // r0: the warp's first row of a block
  // ENV: a factor has no entry further than L.reach points from its diagonal: a warp's eight rows start at the first
  // column its first row couples to and (backward) its eight columns end at the last row its last column
  // couples to, in steps of the four columns that the lanes of a row take together.  Predicated lanes would
  // still occupy the FP64 pipe, so the bounds are the warp's.  The block that a bound cuts stands outside the loop
  // over whole blocks, whose loads can then be issued ahead.
  const int K = L.fd_K.d;
  // forward: y_I = inv(L_II) (rhs_I - sum_{J<I} L_IJ y_J)
  for (int I = 0; I < NB; ++I) {
    const CT* rowblk = F + (size_t)(I * (I + 1) / 2) * 256;
    const int c0 = ENV ? max((fdiv(I * LA_BLK + r0, L.fd_K) - L.reach) * K, 0) >> 2 : 0;   // first group of four columns
    CT acc0 = mkc<CT>(0, 0), acc1 = mkc<CT>(0, 0);
    if (ENV && (c0 & 3) && (c0 >> 2) < I) {
      const CT* blk = rowblk + (c0 >> 2) * 256 + r * LA_BLK;
      const CT* yy = y + (c0 >> 2) * LA_BLK;
      if ((c0 & 3) <= 1) cfma(acc1, blk[l + 4], yy[l + 4]);
      if ((c0 & 3) <= 2) cfma(acc0, blk[l + 8], yy[l + 8]);
      cfma(acc1, blk[l + 12], yy[l + 12]);
    }
    for (int J = (c0 + 3) >> 2; J < I; ++J) {
      const CT* blk = rowblk + J * 256 + r * LA_BLK;
      const CT* yy = y + J * LA_BLK;
      cfma(acc0, blk[l], yy[l]);
      cfma(acc1, blk[l + 4], yy[l + 4]);
      cfma(acc0, blk[l + 8], yy[l + 8]);
      cfma(acc1, blk[l + 12], yy[l + 12]);
    }
    CT acc = reduce4(mkc<CT>(acc0.x + acc1.x, acc0.y + acc1.y));
    if (l == 0) tvec[r] = mkc<CT>(rhs[I * LA_BLK + r].x - acc.x, rhs[I * LA_BLK + r].y - acc.y);
    solve_bar();
    const CT* dblk = rowblk + I * 256 + r * LA_BLK;
    acc0 = mkc<CT>(0, 0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = l + 4 * k;
      if (ENV && 4 * k > r0 + 7) break;
      if (c <= r) cfma(acc0, dblk[c], tvec[c]);
    }
    acc = reduce4(acc0);
    if (l == 0) y[I * LA_BLK + r] = acc;
    solve_bar();
  }
  // backward: x_I = inv(L_II)^dagger (y_I - sum_{J>I} L_JI^dagger x_J), x stored in rhs
  for (int I = NB - 1; I >= 0; --I) {
    const int e4 =   // last group of rows
        (ENV ? min((fdiv(I * LA_BLK + r0 + 7, L.fd_K) + L.reach + 1) * K - 1, NPAD - 1) : NPAD - 1) >> 2;
    CT acc0 = mkc<CT>(0, 0), acc1 = mkc<CT>(0, 0);
    const int Jf = (e4 + 1) >> 2, k1 = (e4 + 1) & 3;   // the first block not taken whole, its groups
    for (int J = I + 1; J < Jf; ++J) {
      const CT* blk = F + (size_t)(J * (J + 1) / 2 + I) * 256;
      const CT* xx = rhs + J * LA_BLK;
      cfma_conj(acc0, blk[l * LA_BLK + r], xx[l]);
      cfma_conj(acc1, blk[(l + 4) * LA_BLK + r], xx[l + 4]);
      cfma_conj(acc0, blk[(l + 8) * LA_BLK + r], xx[l + 8]);
      cfma_conj(acc1, blk[(l + 12) * LA_BLK + r], xx[l + 12]);
    }
    if (ENV && k1 && Jf > I) {
      const CT* blk = F + (size_t)(Jf * (Jf + 1) / 2 + I) * 256;
      const CT* xx = rhs + Jf * LA_BLK;
      cfma_conj(acc0, blk[l * LA_BLK + r], xx[l]);
      if (k1 >= 2) cfma_conj(acc1, blk[(l + 4) * LA_BLK + r], xx[l + 4]);
      if (k1 >= 3) cfma_conj(acc0, blk[(l + 8) * LA_BLK + r], xx[l + 8]);
    }
    CT acc = reduce4(mkc<CT>(acc0.x + acc1.x, acc0.y + acc1.y));
    if (l == 0) tvec[r] = mkc<CT>(y[I * LA_BLK + r].x - acc.x, y[I * LA_BLK + r].y - acc.y);
    solve_bar();
    const CT* dblk = F + (size_t)(I * (I + 1) / 2 + I) * 256;
    acc0 = mkc<CT>(0, 0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int cc = l + 4 * k;
      if (ENV && 4 * k + 3 < r0) continue;
      if (cc >= r) cfma_conj(acc0, dblk[cc * LA_BLK + r], tvec[cc]);
    }
    acc = reduce4(acc0);
    if (l == 0) rhs[I * LA_BLK + r] = acc;
    solve_bar();
  }
}

template <typename CT, int NPAD>
__device__ __forceinline__ void subvol_solve(const LevelGeom& L, const CT* __restrict__ F, CT* rhs, CT* y, CT* tvec) {
  if (solve_inside_envelope(L.reach, L.sub[0] * L.sub[1] * L.sub[2], NPAD / LA_BLK, gridDim.x, sizeof(CT) == 16))
    subvol_solve_t<CT, NPAD, true>(L, F, rhs, y, tvec);
  else subvol_solve_t<CT, NPAD, false>(L, F, rhs, y, tvec);
}

// Triangular solves with a wide factor (more than eight block rows) by all 128 threads of the
// sweep's CTA: every load of a step (one block row forward, one block column backward) is issued
// together, and in complex64 the next step's blocks are loaded while the current step computes, so
// the 2 NB dependent steps wait on memory about once each instead of once per block.  Forward, thread
// (r, q) = (t / 8, t % 8) takes entries (r, 2q) and (r, 2q + 1) of each block of the row (coalesced
// 16-byte pairs); backward, thread (r, q) = (t % 16, t / 16) takes entries (2q, r) and (2q + 1, r) of
// each block of the column (two coalesced rows per warp).  x = (L L^dagger)^{-1} rhs; rhs is
// overwritten by x.  Called by all threads of the CTA, between barriers.
// the two complex entries (2q, r) and (2q + 1, r) of a block (a column pair, stride 16)
template <typename CT>
__device__ __forceinline__ CPair<CT> load_colpair(const CT* blk, int q, int r, unsigned long long pol);
template <>
__device__ __forceinline__ CPair<float2> load_colpair<float2>(const float2* blk, int q, int r, unsigned long long pol) {
  CPair<float2> p;
  const float2 x = ldg_policy(blk + (2 * q) * LA_BLK + r, pol), y = ldg_policy(blk + (2 * q + 1) * LA_BLK + r, pol);
  p.v = make_float4(x.x, x.y, y.x, y.y);
  return p;
}
template <>
__device__ __forceinline__ CPair<double2> load_colpair<double2>(const double2* blk, int q, int r, unsigned long long) {
  CPair<double2> p;
  p.a_ = __ldg(blk + (2 * q) * LA_BLK + r);
  p.b_ = __ldg(blk + (2 * q + 1) * LA_BLK + r);
  return p;
}

template <typename CT>
__device__ __forceinline__ CT reduce_xor(CT v, int m) {
  v.x += __shfl_xor_sync(0xffffffffu, v.x, m);
  v.y += __shfl_xor_sync(0xffffffffu, v.y, m);
  return v;
}

// forward block loads of the solve: complex64 with the keep-for-the-backward-pass policy
template <typename CT>
__device__ __forceinline__ void load_fwd(CPair<CT>& p, const CT* a, unsigned long long pol) {
  p.load(a);
}
template <>
__device__ __forceinline__ void load_fwd<float2>(CPair<float2>& p, const float2* a, unsigned long long pol) {
  p.v = ldg_policy(reinterpret_cast<const float4*>(a), pol);
}
template <typename CT>
__device__ __forceinline__ CPair<CT> zero_pair() {
  CPair<CT> p;
  p.load_zero();
  return p;
}
// a block entry pair inside the band, else the zero it is known to be
template <typename CT>
__device__ __forceinline__ void load_fwd_band(CPair<CT>& p, const CT* a, bool in_band, unsigned long long pol) {
  if (in_band) load_fwd(p, a, pol);
  else p.load_zero();
}

// Whether an FP64 solve leaves the products of zero blocks out (SKIP).  Worth it where the FP64 pipe is the bound and
// enough products go; its branches keep loads from being issued ahead, which costs more where a CTA has an SM for
// itself, and is all there is to it in a wide band.  One colour, every product / without the zero blocks':
//   band 8 of 16 (4x4x4 x 4): 150 CTAs 147 / 168 us, 160 215 / 204 us, 294 220 / 217 us, 343 318 / 280 us, 512 467 / 449 us;
//   band 4 (8x8 x 4): 160 CTAs 199 / 142 us, 400 295 / 197 us (100: 128 / 114 us, but 16x4 x 4 131 / 147 us);
//   band 7 of 12 (4x4x4 x 3): 160 CTAs 136 / 135 us, 294 140 / 142 us, 343 200 / 186 us;
//   band 11 of 16 (4x4x3 x 5): 160 CTAs 221 / 232 us, 343 414 / 456 us; band 15 (8x4x2 x 4): 343 CTAs 409 / 471 us.
template <int NB>
__device__ __forceinline__ bool skip_zero_blocks(int band, unsigned ctas) {
  return 2 * band <= NB ? ctas > kSms : 3 * band <= 2 * NB && ctas > 2 * kSms;
}
template <typename CT, int NPAD, bool SKIP>
__device__ __forceinline__ void subvol_solve_wide(const CT* __restrict__ F, int band, CT* rhs, CT* y, CT* tvec,
                                                  CT* part) {
  constexpr int NB = NPAD / LA_BLK;
  constexpr bool kPrefetch = sizeof(CT) == 8;   // complex64: next step's blocks in flight during this one
  const int t = threadIdx.x;
  const unsigned long long keep = l2_evict_last(), last_use = l2_evict_first();
  {
    const int r = t >> 3, q = t & 7;
    CPair<CT> cur[NB];
    load_fwd(cur[0], F + r * LA_BLK + 2 * q, keep);
#pragma unroll
    for (int I = 0; I < NB; ++I) {
      CPair<CT> nxt[NB];
      // blocks (I, J) with I - J > band are exact zeros: set, not loaded
      if (kPrefetch && I + 1 < NB) {
#pragma unroll
        for (int J = 0; J <= I + 1; ++J)
          load_fwd_band(nxt[J], F + (size_t)tri_index(I + 1, J) * 256 + r * LA_BLK + 2 * q, J >= I + 1 - band, keep);
      }
      if (!kPrefetch && I > 0) {
#pragma unroll
        for (int J = 0; J <= I; ++J)
          load_fwd_band(cur[J], F + (size_t)tri_index(I, J) * 256 + r * LA_BLK + 2 * q, J >= I - band, keep);
      }
      CT acc0 = mkc<CT>(0, 0), acc1 = mkc<CT>(0, 0);
#pragma unroll
      for (int J = 0; J < I; ++J) {
        if (SKIP && J < I - band) continue;   // zero blocks: their products would still take the pipe
        cfma(acc0, cur[J].a(), y[J * LA_BLK + 2 * q]);
        cfma(acc1, cur[J].b(), y[J * LA_BLK + 2 * q + 1]);
      }
      CT acc = mkc<CT>(acc0.x + acc1.x, acc0.y + acc1.y);
      acc = reduce_xor(acc, 1);
      acc = reduce_xor(acc, 2);
      acc = reduce_xor(acc, 4);
      if (q == 0) tvec[r] = mkc<CT>(rhs[I * LA_BLK + r].x - acc.x, rhs[I * LA_BLK + r].y - acc.y);
      __syncthreads();
      CT d = mkc<CT>(0, 0);
      cfma(d, cur[I].a(), tvec[2 * q]);
      cfma(d, cur[I].b(), tvec[2 * q + 1]);
      d = reduce_xor(d, 1);
      d = reduce_xor(d, 2);
      d = reduce_xor(d, 4);
      if (q == 0) y[I * LA_BLK + r] = d;
      __syncthreads();
      if (kPrefetch) {
#pragma unroll
        for (int J = 0; J < NB; ++J) cur[J] = nxt[J];
      }
    }
  }
  {
    const int r = t & 15, q = t >> 4, w = t >> 5;
    CPair<CT> cur[NB];
    // step I uses blocks (J, I), J = I .. NB-1 ((I, I): the inverted diagonal block)
    if (kPrefetch) {
#pragma unroll
      for (int J = NB - 1; J < NB; ++J) cur[J] = load_colpair<CT>(F + (size_t)tri_index(J, NB - 1) * 256, q, r, last_use);
    }
#pragma unroll
    for (int I = NB - 1; I >= 0; --I) {
      CPair<CT> nxt[NB];
      if (kPrefetch && I > 0) {
#pragma unroll
        for (int J = I - 1; J < NB; ++J)
          nxt[J] = J <= I - 1 + band ? load_colpair<CT>(F + (size_t)tri_index(J, I - 1) * 256, q, r, last_use)
                                     : zero_pair<CT>();
      }
      if (!kPrefetch) {
#pragma unroll
        for (int J = I; J < NB; ++J)
          cur[J] = J <= I + band ? load_colpair<CT>(F + (size_t)tri_index(J, I) * 256, q, r, last_use) : zero_pair<CT>();
      }
      CT acc0 = mkc<CT>(0, 0), acc1 = mkc<CT>(0, 0);
#pragma unroll
      for (int J = I + 1; J < NB; ++J) {
        if (SKIP && J > I + band) continue;
        cfma_conj(acc0, cur[J].a(), rhs[J * LA_BLK + 2 * q]);
        cfma_conj(acc1, cur[J].b(), rhs[J * LA_BLK + 2 * q + 1]);
      }
      CT acc = reduce_xor(mkc<CT>(acc0.x + acc1.x, acc0.y + acc1.y), 16);
      if ((t & 16) == 0) part[w * LA_BLK + r] = acc;
      __syncthreads();
      if (t < LA_BLK) {
        CT s = part[r];
#pragma unroll
        for (int u = 1; u < 4; ++u) { s.x += part[u * LA_BLK + r].x; s.y += part[u * LA_BLK + r].y; }
        tvec[r] = mkc<CT>(y[I * LA_BLK + r].x - s.x, y[I * LA_BLK + r].y - s.y);
      }
      __syncthreads();
      CT d = mkc<CT>(0, 0);
      cfma_conj(d, cur[I].a(), tvec[2 * q]);
      cfma_conj(d, cur[I].b(), tvec[2 * q + 1]);
      d = reduce_xor(d, 16);
      if ((t & 16) == 0) part[w * LA_BLK + r] = d;
      __syncthreads();
      if (t < LA_BLK) {
        CT s = part[r];
#pragma unroll
        for (int u = 1; u < 4; ++u) { s.x += part[u * LA_BLK + r].x; s.y += part[u * LA_BLK + r].y; }
        rhs[I * LA_BLK + r] = s;
      }
      __syncthreads();
      if (kPrefetch) {
#pragma unroll
        for (int J = 0; J < NB; ++J) cur[J] = nxt[J];
      }
    }
  }
}

// Solves with a factor whose diagonal superblocks hold inverses (factor_is_super), by 256 threads.  With
// 64-row superblocks R: forward t_R = rhs_R - sum_{C<R} L_RC y_C, y_R = X_RR t_R; backward
// t_R = y_R - sum_{C>R} L_CR^dagger x_C, x_R = X_RR^dagger t_R: 2 NB / 4 steps of two mat-vecs each instead of
// 2 NB steps of 16 rows, so a subvolume's chain is 14 barriers.  A mat-vec runs through its 16 x 16 blocks
// in pieces of four 16-byte loads per lane, issued kAhead pieces before they are used.
// What bounds it is the L1 data path (the factor passes through it twice), so the vectors must cost little
// there: forward, warp (i, half) = (w / 2, w % 2) takes the blocks of block row i with even or odd column and
// lane (row l / 8, column pair l % 8) four rows of a block, so that one 16-byte vector load serves a block;
// the halves' sums stay apart in shared memory and are added by whoever reads them.  Backward, warp w takes
// columns 8 w .. + 7, lane (row l / 4, column pair l % 4) two rows of a block.
struct SuperPiece {
  float4 v[4];
};
__device__ __forceinline__ float4 ldg_block(const float2* p, bool valid, unsigned long long pol) {
  return valid ? ldg_policy(reinterpret_cast<const float4*>(p), pol) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) {
  return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float2 shfl_xor2(float2 v, int m) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
// One exchange of a transposing reduction: lanes without bit m of their index keep a, the others b, each
// adding the partner's share.
__device__ __forceinline__ float2 fold(float2 a, float2 b, bool hi, int m) {
  const float2 send = hi ? a : b, mine = hi ? b : a, got = shfl_xor2(send, m);
  return make_float2(mine.x + got.x, mine.y + got.y);
}

// rhs [NPAD] in; the solution goes to x [NPAD].  y [2][NPAD], p [2][64]: scratch, the halves' sums.
template <int NPAD>
__device__ __forceinline__ void subvol_solve_super(const float2* __restrict__ F, int band, const float2* rhs, float2* y,
                                                   float2* p, float2* x) {
  constexpr int NS = NPAD / (LA_BLK * kSuper);
  // pieces of the forward pass: rows R = 0 .. NS-1, columns C = 0 .. R, two each; the backward pass takes the
  // transposed ones, rows NS-1 .. 0
  constexpr int NP = NS * (NS + 1);
  constexpr int kAhead = 1, NBUF = kAhead + 1;
  const int tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  const unsigned long long keep = l2_evict_last(), last_use = l2_evict_first();
  const int bi = w >> 1, wh = w & 1;     // block row (forward) or column (backward) in the superblock, half
  const int fq = l & 7, fr = l >> 3, bq = l & 3, br = l >> 2;
  const float2* const fbase = F + (size_t)(bi * (bi + 1) / 2 + wh) * 256 + fr * LA_BLK + 2 * fq;
  const float2* const bbase = F + (size_t)bi * 256 + br * LA_BLK + 8 * wh + 2 * bq;
  auto row_of = [](int s) constexpr {
    int R = 0;
    while ((R + 1) * (R + 2) <= s) ++R;
    return R;
  };
  auto fwd_ok = [&](int R, int C, int jj) { return R == C ? jj <= bi : kSuper * (R - C) + bi - jj <= band; };
  auto bwd_ok = [&](int C, int R, int ii) { return R == C ? ii >= bi : kSuper * (C - R) + ii - bi <= band; };
  SuperPiece buf[NBUF];
  auto load = [&](SuperPiece& b, int s) {   // piece s of both passes, 0 .. 2 NP - 1
    const int q = s < NP ? s : s - NP;
    const int A = row_of(q), B = (q - A * (A + 1)) >> 1, h = (q - A * (A + 1)) & 1;
    if (s < NP) {   // block (4 A + bi, 4 B + 2 h + wh); tri_index(4 A + i, J) = 8 A^2 + 2 A + 4 A i + tri(i) + J
      const float2* a = fbase + (size_t)(4 * A * bi) * 256 + (8 * A * A + 2 * A + kSuper * B + 2 * h) * 256;
      const bool ok = fwd_ok(A, B, 2 * h + wh);
#pragma unroll
      for (int u = 0; u < 4; ++u) b.v[u] = ldg_block(a + 4 * u * LA_BLK, ok, keep);
    } else {   // blocks (4 C + 2 h, 4 C + 2 h + 1) of columns R = NS-1-A, C = NS-1-B
      const int R = NS - 1 - A, C = NS - 1 - B;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int ii = 2 * h + u, I = kSuper * C + ii;
        const float2* a = bbase + (size_t)(I * (I + 1) / 2 + kSuper * R) * 256;
        const bool ok = bwd_ok(C, R, ii);
        b.v[2 * u] = ldg_block(a, ok, last_use);
        b.v[2 * u + 1] = ldg_block(a + 8 * LA_BLK, ok, last_use);
      }
    }
  };
#pragma unroll
  for (int s = 0; s < kAhead; ++s) load(buf[s], s);
  const float2 zero = make_float2(0.f, 0.f);
  float2 acc[4] = {zero, zero, zero, zero};
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const int R = row_of(s), C = (s - R * (R + 1)) >> 1, h = (s - R * (R + 1)) & 1;
    load(buf[(s + kAhead) % NBUF], s + kAhead);
    const SuperPiece& b = buf[s % NBUF];
    const int jj = 2 * h + wh;
    if (fwd_ok(R, C, jj)) {
      const int at = LA_BLK * jj + 2 * fq;
      float4 v;
      if (C < R) {
        v = add4(*reinterpret_cast<const float4*>(y + 64 * C + at), *reinterpret_cast<const float4*>(y + NPAD + 64 * C + at));
      } else {
        v = *reinterpret_cast<const float4*>(rhs + 64 * R + at);
        if (R > 0) v = sub4(sub4(v, *reinterpret_cast<const float4*>(p + at)), *reinterpret_cast<const float4*>(p + 64 + at));
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        cfma(acc[u], make_float2(b.v[u].x, b.v[u].y), make_float2(v.x, v.y));
        cfma(acc[u], make_float2(b.v[u].z, b.v[u].w), make_float2(v.z, v.w));
      }
    }
    if (h == 1 && (C == R || C == R - 1)) {
      // the four rows over the eight column pairs: lane fq ends with row fr + 4 (fq / 2)
      const float2 a = fold(acc[0], acc[2], fq & 4, 4), c = fold(acc[1], acc[3], fq & 4, 4);
      float2 r = fold(a, c, fq & 2, 2);
      r = reduce_xor(r, 1);
      if (!(fq & 1)) (C == R ? y + wh * NPAD + 64 * R : p + 64 * wh)[LA_BLK * bi + fr + 4 * (fq >> 1)] = r;
      acc[0] = acc[1] = acc[2] = acc[3] = zero;
      __syncthreads();
    }
  }
  float2 acc0 = zero, acc1 = zero;
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    const int A = row_of(s), R = NS - 1 - A, C = NS - 1 - ((s - A * (A + 1)) >> 1), h = (s - A * (A + 1)) & 1;
    if (s + kAhead < NP) load(buf[(NP + s + kAhead) % NBUF], NP + s + kAhead);
    const SuperPiece& b = buf[(NP + s) % NBUF];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int ii = 2 * h + u;
      if (!bwd_ok(C, R, ii)) continue;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int row = LA_BLK * ii + br + 8 * e;
        float2 v;
        if (C > R) {
          v = x[64 * C + row];
        } else {
          const float2 y0 = y[64 * R + row], y1 = y[NPAD + 64 * R + row];
          v = make_float2(y0.x + y1.x, y0.y + y1.y);
          if (R < NS - 1) {
            const float2 q = p[row];
            v = make_float2(v.x - q.x, v.y - q.y);
          }
        }
        const float4 m = b.v[2 * u + e];
        cfma_conj(acc0, make_float2(m.x, m.y), v);
        cfma_conj(acc1, make_float2(m.z, m.w), v);
      }
    }
    if (h == 1 && (C == R || C == R + 1)) {
      float2 r = fold(acc0, acc1, br & 1, 4);
      r = reduce_xor(r, 8);
      r = reduce_xor(r, 16);
      if (br < 2) (C == R ? x + 64 * R : p)[8 * w + 2 * bq + br] = r;
      acc0 = acc1 = zero;
      __syncthreads();
    }
  }
}

// Solves with the stored inverse X = inv(L) of a complex64 factor of at most 32 unknowns (factor_is_inverse):
// y = X rhs, x = X^dagger y, two mat-vecs by 128 threads instead of four block steps with eight barriers.  The
// factor's entries (at most seven 16-byte loads per thread) are loaded before the right-hand side is formed.
// Forward, thread (row t / 4, quarter t % 4) takes four columns of each block; backward, thread (row t / 8,
// column pair t % 8) one row of each block; the four warps' sums are added by the caller, x_i = sum_w part[32 w + i].
template <int NPAD>
struct InverseFactor {
  static constexpr int NB = NPAD / LA_BLK;
  float4 f[2 * NB], b[2 * NB - 1];
  __device__ __forceinline__ void load(const float2* __restrict__ F) {
    const int t = threadIdx.x, r = t >> 2, q = t & 3, rr = t >> 3, q8 = t & 7;
    const bool row = r < NPAD;
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        f[2 * J + u] = row && J <= (r >> 4)
                           ? __ldg(reinterpret_cast<const float4*>(F + tri_index(r >> 4, J) * 256 + (r & 15) * LA_BLK + 4 * q + 2 * u))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 2 * NB - 1; ++u)   // blocks (0,0), (1,0), (1,1)
      b[u] = __ldg(reinterpret_cast<const float4*>(F + u * 256 + rr * LA_BLK + 2 * q8));
  }
  __device__ __forceinline__ void solve(const float2* rhs, float2* y, float2* part) const {
    const int t = threadIdx.x, r = t >> 2, q = t & 3, l = t & 31, rr = t >> 3, q8 = t & 7;
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float2* x = rhs + LA_BLK * J + 4 * q + 2 * u;
        cfma(a0, make_float2(f[2 * J + u].x, f[2 * J + u].y), x[0]);
        cfma(a1, make_float2(f[2 * J + u].z, f[2 * J + u].w), x[1]);
      }
    float2 a = make_float2(a0.x + a1.x, a0.y + a1.y);
    a = reduce_xor(a, 1);
    a = reduce_xor(a, 2);
    if (q == 0 && r < NPAD) y[r] = a;
    __syncthreads();
    // columns 2 q8, 2 q8 + 1 of block column 0 (c0, c1) and 1 (c2, c3)
    float2 c0 = make_float2(0.f, 0.f), c1 = c0, c2 = c0, c3 = c0;
    const float2 y0 = y[rr];
    cfma_conj(c0, make_float2(b[0].x, b[0].y), y0);
    cfma_conj(c1, make_float2(b[0].z, b[0].w), y0);
    if (NB > 1) {
      const float2 y1 = y[LA_BLK + rr];
      cfma_conj(c0, make_float2(b[2 * NB - 3 > 0 ? 1 : 0].x, b[2 * NB - 3 > 0 ? 1 : 0].y), y1);
      cfma_conj(c1, make_float2(b[2 * NB - 3 > 0 ? 1 : 0].z, b[2 * NB - 3 > 0 ? 1 : 0].w), y1);
      cfma_conj(c2, make_float2(b[2 * NB - 2].x, b[2 * NB - 2].y), y1);
      cfma_conj(c3, make_float2(b[2 * NB - 2].z, b[2 * NB - 2].w), y1);
    }
    // over the warp's four rows (lane bits 3, 4): lane (bit 3, bit 4) ends with column 2 q8 + bit 3 of block bit 4
    float2 s = fold(c0, c1, l & 8, 8);
    if (NB > 1) s = fold(s, fold(c2, c3, l & 8, 8), l & 16, 16);
    else s = reduce_xor(s, 16);
    if (NB > 1 || !(l & 16)) part[(t & ~31) + ((l & 16) ? LA_BLK : 0) + 2 * q8 + ((l >> 3) & 1)] = s;
    __syncthreads();
  }
  __device__ __forceinline__ static float2 result(const float2* part, int i) {
    float2 s = part[i];
#pragma unroll
    for (int w = 1; w < 4; ++w) { s.x += part[32 * w + i].x; s.y += part[32 * w + i].y; }
    return s;
  }
};
// complex64 factors of at most 32 unknowns are stored as the inverse of L (k_factor_small).
template <typename R, int NPAD>
__host__ __device__ constexpr bool factor_is_inverse() {
  return sizeof(R) == 4 && NPAD <= 32;
}
template <typename R, int NPAD, bool ON> struct MaybeInverse {};
template <typename R, int NPAD> struct MaybeInverse<R, NPAD, true> : InverseFactor<NPAD> {};

// The 128-thread solve (every step's blocks loaded together, the next step's in flight) serves every
// complex64 factor and the wide FP64 ones; shorter FP64 factors keep the two-warp solve, whose
// two-level reductions issue fewer adds on the slow FP64 pipe.
template <typename R, int NPAD>
__host__ __device__ constexpr bool use_wide_solve() {
  return sizeof(R) == 4 || NPAD > LA_NPAD_MAX;
}

// ======================================================================== finest-level sweep
// Matrix-free (M-form): residual r = f - M~ c on the footprint F = U + 1 from c on U + 2,
// z = Wt r, right-hand side (M~^dagger z)_U, solve, c_U += delta.
template <typename R, int NPAD>
__global__ void __launch_bounds__(kSweepThreads)
k_sweep_fine(LevelGeom L, FineOp g, const TimeMats* __restrict__ tm, const typename C2<R>::T* f,
             const typename C2<R>::T* yx, typename C2<R>::T* c, const typename C2<R>::T* __restrict__ factors,
             int colour) {
  typedef typename C2<R>::T CT;
  extern __shared__ __align__(16) unsigned char smem[];
  overlap_trigger();
  const int K = tm->K, KK = K * K;
  const int tid = threadIdx.x;
  const int b = colour_subvol(L, colour, blockIdx.x);
  int o[3], e[3];
  subvol_box(L, b, o, e);
  int ec[3], ef[3], oc[3], of_[3];
  for (int a = 0; a < 3; ++a) {
    const bool used = a < L.dim;
    ec[a] = used ? e[a] + 4 : 1;  oc[a] = used ? o[a] - 2 : o[a];
    ef[a] = used ? e[a] + 2 : 1;  of_[a] = used ? o[a] - 1 : o[a];
  }
  const int nbc = ec[0] * ec[1] * ec[2], nbf = ef[0] * ef[1] * ef[2], npts = e[0] * e[1] * e[2];
  const int sx = L.sub[0] + 4, sy = L.dim > 1 ? L.sub[1] + 4 : 1, sz = L.dim > 2 ? L.sub[2] + 4 : 1;
  const int nbc_max = sx * sy * sz;
  const int nbf_max = (L.sub[0] + 2) * (L.dim > 1 ? L.sub[1] + 2 : 1) * (L.dim > 2 ? L.sub[2] + 2 : 1);
  // index maps item t -> (point i, time function m) and point -> (x, y, z) by multiply-shift
  // division: the level's divisors for a full subvolume, this CTA's own for a ragged one
  const bool full = e[0] == L.sub[0] && e[1] == L.sub[1] && e[2] == L.sub[2];
  const FastDiv dK = L.fd_K;
  const FastDiv dc0 = full ? L.fd_c[0] : make_fastdiv(ec[0]), dc1 = full ? L.fd_c[1] : make_fastdiv(ec[1]);
  const FastDiv df0 = full ? L.fd_f[0] : make_fastdiv(ef[0]), df1 = full ? L.fd_f[1] : make_fastdiv(ef[1]);
  const FastDiv du0 = full ? L.fd_u[0] : make_fastdiv(e[0]), du1 = full ? L.fd_u[1] : make_fastdiv(e[1]);
  auto item = [&](int t, int& i, int& m) {
    i = fdiv(t, dK);
    m = t - i * K;
  };
  auto coords = [](int i, const FastDiv& d0, const FastDiv& d1, int& x, int& y, int& z) {
    const int r = fdiv(i, d0);
    x = i - r * d0.d;
    z = fdiv(r, d1);
    y = r - z * d1.d;
  };

  R* sQ = reinterpret_cast<R*>(smem);
  R* sU = sQ + LA_KMAX * LA_KMAX;
  R* sW = sU + LA_KMAX * LA_KMAX;
  R* sE = sW + LA_KMAX * LA_KMAX;
  R* sV = sE + LA_KMAX * LA_KMAX;                     // dsum + V0 on the footprint F = U + 1 [nbf_max]
  R* sX = sV + ((nbf_max + 3) & ~3);                  // laser coordinate on the footprint [nbf_max]
  CT* sC = reinterpret_cast<CT*>(sX + ((nbf_max + 3) & ~3));  // c on U+2  [nbc_max * K]
  CT* sA = sC + (size_t)nbc_max * K;                  // Hc, then z, on the footprint   [nbf_max * K]
  CT* sB = sA + (size_t)nbf_max * K;                  // r, then Hz, on the footprint   [nbf_max * K]
  CT* sRhs = sB + (size_t)nbf_max * K;                // [NPAD]
  CT* sY = sRhs + NPAD;                               // [NPAD]
  CT* sT = sY + NPAD;                                 // [16]
  CT* sRed = sT + LA_BLK;                             // [128]

  for (int i = tid; i < KK; i += kSweepThreads) {
    sQ[i] = (R)tm->Qb[i]; sU[i] = (R)tm->Ub[i]; sW[i] = (R)tm->Wt[i]; sE[i] = (R)tm->Eb[i];
  }
  overlap_wait();
  const unsigned long long stream = l2_evict_first();   // c and f: read once per launch
  for (int t = tid; t < nbc * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    int lx, ly, lz;
    coords(i, dc0, dc1, lx, ly, lz);
    const int gx = oc[0] + lx, gy = oc[1] + ly, gz = oc[2] + lz;
    CT v = mkc<CT>(0, 0);
    if (fine_in(g, gx, gy, gz)) v = ld_policy(c + (size_t)((gz * g.n[1] + gy) * g.n[0] + gx) * K + m, stream);
    sC[t] = v;
  }
  {
    // per footprint point, in the kernel's own precision (a complex64 sweep issues no FP64 work here)
    const R dsum = (R)g.dsum;
    const R xo = (R)(g.lax == 0 ? g.x0[0] : (g.lax == 1 ? g.x0[1] : g.x0[2]));
    const R xh = (R)(g.lax == 0 ? g.h[0] : (g.lax == 1 ? g.h[1] : g.h[2]));
    for (int i = tid; i < nbf; i += kSweepThreads) {
      int lx, ly, lz;
      coords(i, df0, df1, lx, ly, lz);
      const int gx = of_[0] + lx, gy = of_[1] + ly, gz = of_[2] + lz;
      sV[i] = fine_in(g, gx, gy, gz) ? dsum + (R)g.V0[(gz * g.n[1] + gy) * g.n[0] + gx] : (R)0;
      sX[i] = xo + (R)(g.lax == 0 ? gx : (g.lax == 1 ? gy : gz)) * xh;
    }
  }
  __syncthreads();
  // c-box index of footprint point (lx, ly, lz): (lx+1, ly+1, lz+1) on used axes
  const int dcx = 1, dcy = L.dim > 1 ? ec[0] : 0, dcz = L.dim > 2 ? ec[0] * ec[1] : 0;
  const R wx = (R)(-0.5 * g.ih2[0]), wy = (R)(-0.5 * g.ih2[1]), wz = (R)(-0.5 * g.ih2[2]);
  // stage 1: Hc on the footprint
  for (int t = tid; t < nbf * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    int lx, ly, lz;
    coords(i, df0, df1, lx, ly, lz);
    const int cx = L.dim > 0 ? lx + 1 : lx, cy = L.dim > 1 ? ly + 1 : ly, cz = L.dim > 2 ? lz + 1 : lz;
    const int ci = (cz * ec[1] + cy) * ec[0] + cx;
    const CT v = sC[ci * K + m];
    CT h = mkc<CT>(sV[i] * v.x, sV[i] * v.y);
    {
      const CT a1 = sC[(ci + dcx) * K + m], a2 = sC[(ci - dcx) * K + m];
      h.x += wx * (a1.x + a2.x); h.y += wx * (a1.y + a2.y);
    }
    if (L.dim > 1) {
      const CT a1 = sC[(ci + dcy) * K + m], a2 = sC[(ci - dcy) * K + m];
      h.x += wy * (a1.x + a2.x); h.y += wy * (a1.y + a2.y);
    }
    if (L.dim > 2) {
      const CT a1 = sC[(ci + dcz) * K + m], a2 = sC[(ci - dcz) * K + m];
      h.x += wz * (a1.x + a2.x); h.y += wz * (a1.y + a2.y);
    }
    sA[t] = h;
  }
  __syncthreads();
  // stage 2: r = f - (i Qb c - Ub Hc - x Eb c) on the footprint (0 outside the grid)
  for (int t = tid; t < nbf * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    int lx, ly, lz;
    coords(i, df0, df1, lx, ly, lz);
    const int gx = of_[0] + lx, gy = of_[1] + ly, gz = of_[2] + lz;
    CT r = mkc<CT>(0, 0);
    if (fine_in(g, gx, gy, gz)) {
      const int cx = L.dim > 0 ? lx + 1 : lx, cy = L.dim > 1 ? ly + 1 : ly, cz = L.dim > 2 ? lz + 1 : lz;
      const int ci = (cz * ec[1] + cy) * ec[0] + cx;
      const R xl = sX[i];
      R qr = 0, qi = 0, ur = 0, ui = 0, er = 0, ei = 0;
      for (int nn = 0; nn < K; ++nn) {
        const CT cv = sC[ci * K + nn], hv = sA[i * K + nn];
        const R q = sQ[m * K + nn], u = sU[m * K + nn], ee = sE[m * K + nn];
        qr = fma(q, cv.x, qr); qi = fma(q, cv.y, qi);
        ur = fma(u, hv.x, ur); ui = fma(u, hv.y, ui);
        er = fma(ee, cv.x, er); ei = fma(ee, cv.y, ei);
      }
      const CT fv = f ? ld_policy(f + (size_t)((gz * g.n[1] + gy) * g.n[0] + gx) * K + m, stream) : mkc<CT>(0, 0);
      r.x = fv.x - (-qi - ur - xl * er);
      r.y = fv.y - (qr - ui - xl * ei);
    }
    sB[t] = r;
  }
  __syncthreads();
  // stage 3: z = Wt r
  for (int t = tid; t < nbf * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    R zr = 0, zi = 0;
    for (int nn = 0; nn < K; ++nn) {
      const R w = sW[m * K + nn];
      const CT rv = sB[i * K + nn];
      zr = fma(w, rv.x, zr); zi = fma(w, rv.y, zi);
    }
    sA[t] = mkc<CT>(zr, zi);
  }
  __syncthreads();
  // stage 4: Hz on U (footprint index of U point = local + 1 on used axes)
  const int dfy = L.dim > 1 ? ef[0] : 0, dfz = L.dim > 2 ? ef[0] * ef[1] : 0;
  for (int t = tid; t < npts * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    int lx, ly, lz;
    coords(i, du0, du1, lx, ly, lz);
    const int fx = L.dim > 0 ? lx + 1 : lx, fy = L.dim > 1 ? ly + 1 : ly, fz = L.dim > 2 ? lz + 1 : lz;
    const int fi = (fz * ef[1] + fy) * ef[0] + fx;
    const CT v = sA[fi * K + m];
    CT h = mkc<CT>(sV[fi] * v.x, sV[fi] * v.y);
    {
      const CT a1 = sA[(fi + 1) * K + m], a2 = sA[(fi - 1) * K + m];
      h.x += wx * (a1.x + a2.x); h.y += wx * (a1.y + a2.y);
    }
    if (L.dim > 1) {
      const CT a1 = sA[(fi + dfy) * K + m], a2 = sA[(fi - dfy) * K + m];
      h.x += wy * (a1.x + a2.x); h.y += wy * (a1.y + a2.y);
    }
    if (L.dim > 2) {
      const CT a1 = sA[(fi + dfz) * K + m], a2 = sA[(fi - dfz) * K + m];
      h.x += wz * (a1.x + a2.x); h.y += wz * (a1.y + a2.y);
    }
    sB[t] = h;
  }
  __syncthreads();
  // stage 5: rhs = -i Qb^T z - Ub Hz - x Eb z on U; padding 0
  for (int t = tid; t < NPAD; t += kSweepThreads) {
    CT out = mkc<CT>(0, 0);
    if (t < npts * K) {
      int i, m;
      item(t, i, m);
      int lx, ly, lz;
      coords(i, du0, du1, lx, ly, lz);
      const int fx = L.dim > 0 ? lx + 1 : lx, fy = L.dim > 1 ? ly + 1 : ly, fz = L.dim > 2 ? lz + 1 : lz;
      const int fi = (fz * ef[1] + fy) * ef[0] + fx;
      const R xl = sX[fi];
      R qr = 0, qi = 0, ur = 0, ui = 0, er = 0, ei = 0;
      for (int nn = 0; nn < K; ++nn) {
        const CT zv = sA[fi * K + nn], hv = sB[i * K + nn];
        const R q = sQ[nn * K + m], u = sU[m * K + nn], ee = sE[m * K + nn];
        qr = fma(q, zv.x, qr); qi = fma(q, zv.y, qi);
        ur = fma(u, hv.x, ur); ui = fma(u, hv.y, ui);
        er = fma(ee, zv.x, er); ei = fma(ee, zv.y, ei);
      }
      out.x = qi - ur - xl * er;
      out.y = -qr - ui - xl * ei;
      if (yx) {  // additive right-hand side (adjoint relaxation of G z = y)
        const CT yv = yx[(size_t)(((o[2] + lz) * g.n[1] + (o[1] + ly)) * g.n[0] + (o[0] + lx)) * K + m];
        out.x += yv.x;
        out.y += yv.y;
      }
    }
    sRhs[t] = out;
  }
  __syncthreads();
  if (use_wide_solve<R, NPAD>()) {
    if (sizeof(R) == 8 && skip_zero_blocks<NPAD / LA_BLK>(L.band, gridDim.x))
      subvol_solve_wide<CT, NPAD, true>(factors + (size_t)b * L.fsize, L.band, sRhs, sY, sT, sRed);
    else
      subvol_solve_wide<CT, NPAD, false>(factors + (size_t)b * L.fsize, L.band, sRhs, sY, sT, sRed);
  } else
    subvol_solve<CT, NPAD>(L, factors + (size_t)b * L.fsize, sRhs, sY, sT);
  __syncthreads();
  for (int t = tid; t < npts * K; t += kSweepThreads) {
    int i, m;
    item(t, i, m);
    int lx, ly, lz;
    coords(i, du0, du1, lx, ly, lz);
    const size_t gi = (size_t)(((o[2] + lz) * g.n[1] + (o[1] + ly)) * g.n[0] + (o[0] + lx)) * K + m;
    CT v = c[gi];
    v.x += sRhs[t].x;
    v.y += sRhs[t].y;
    c[gi] = v;
  }
}

// Shared memory of k_sweep_super: byte offsets of its arrays (the time matrices are at 0) and the total.
struct SuperSmem {
  int v, c, z, rhs, total;
};
__host__ __device__ __forceinline__ SuperSmem super_smem(const LevelGeom& L, int K) {
  const int nbc = (L.sub[0] + 4) * (L.dim > 1 ? L.sub[1] + 4 : 1) * (L.dim > 2 ? L.sub[2] + 4 : 1);
  const int nbf = (L.sub[0] + 2) * (L.dim > 1 ? L.sub[1] + 2 : 1) * (L.dim > 2 ? L.sub[2] + 2 : 1);
  SuperSmem s;
  s.v = (5 * K * K * 4 + 15) & ~15;
  s.c = s.v + ((nbf * 4 + 15) & ~15);
  s.z = s.c + ((nbc * K * 8 + 15) & ~15);
  s.rhs = s.z + ((nbf * K * 8 + 15) & ~15);
  s.total = s.rhs + (4 * L.npad + 128) * 8;   // rhs, the solution, y in two halves, products in two halves
  return s;
}

// ------------------------------------------------------------------------ finest sweep, superblock factors
// Rows of K floats of the time matrices from shared memory, in the widest loads K allows.
template <int K>
__device__ __forceinline__ void row_k(const float* p, float (&r)[K]) {
  if constexpr (K % 4 == 0) {
#pragma unroll
    for (int n = 0; n < K; n += 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + n);
      r[n] = v.x; r[n + 1] = v.y; r[n + 2] = v.z; r[n + 3] = v.w;
    }
  } else if constexpr (K % 2 == 0) {
#pragma unroll
    for (int n = 0; n < K; n += 2) {
      const float2 v = *reinterpret_cast<const float2*>(p + n);
      r[n] = v.x; r[n + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int n = 0; n < K; ++n) r[n] = p[n];
  }
}
// The K complex values of a point's record.
template <int K>
__device__ __forceinline__ void rec_k(const float2* p, float2 (&v)[K]) {
  if constexpr (K % 2 == 0) {
#pragma unroll
    for (int n = 0; n < K; n += 2) {
      const float4 q = *reinterpret_cast<const float4*>(p + n);
      v[n] = make_float2(q.x, q.y);
      v[n + 1] = make_float2(q.z, q.w);
    }
  } else {
#pragma unroll
    for (int n = 0; n < K; ++n) v[n] = p[n];
  }
}

// Geometry of one subvolume of a colour for the point-per-thread right-hand side: origin and extent of U, of
// U + 1 (footprint) and of U + 2 (c box), and the multiply-shift divisors of their index maps (the level's for
// a full subvolume, its own for a ragged one).
struct SweepBox {
  int o[3], e[3], ec[3], ef[3], oc[3], of_[3];
  FastDiv dc0, dc1, df0, df1, du0, du1;
  // j-th subvolume of the colour; dn0, dn1 divide by the colour's subvolumes along x and y.  Returns its index.
  __device__ __forceinline__ int init(const LevelGeom& L, int colour, int j, const FastDiv& dn0, const FastDiv& dn1) {
    const int jr = fdiv(j, dn0), jz = fdiv(jr, dn1);
    const int bb[3] = {2 * (j - jr * dn0.d) + (colour & 1), 2 * (jr - jz * dn1.d) + ((colour >> 1) & 1),
                       2 * jz + ((colour >> 2) & 1)};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const bool used = a < L.dim;
      o[a] = bb[a] * L.sub[a];
      e[a] = min(L.sub[a], L.n[a] - o[a]);
      ec[a] = used ? e[a] + 4 : 1;  oc[a] = used ? o[a] - 2 : o[a];
      ef[a] = used ? e[a] + 2 : 1;  of_[a] = used ? o[a] - 1 : o[a];
    }
    const bool full = e[0] == L.sub[0] && e[1] == L.sub[1] && e[2] == L.sub[2];
    dc0 = full ? L.fd_c[0] : make_fastdiv(ec[0]);  dc1 = full ? L.fd_c[1] : make_fastdiv(ec[1]);
    df0 = full ? L.fd_f[0] : make_fastdiv(ef[0]);  df1 = full ? L.fd_f[1] : make_fastdiv(ef[1]);
    du0 = full ? L.fd_u[0] : make_fastdiv(e[0]);   du1 = full ? L.fd_u[1] : make_fastdiv(e[1]);
    return (bb[2] * L.nb[1] + bb[1]) * L.nb[0] + bb[0];
  }
  __device__ __forceinline__ static void coords(int i, const FastDiv& d0, const FastDiv& d1, int& x, int& y, int& z) {
    const int r = fdiv(i, d0);
    x = i - r * d0.d;
    z = fdiv(r, d1);
    y = r - z * d1.d;
  }
};
// The time matrices in complex64 as the right-hand side reads them: Q, U, E, W, Q^T, K x K floats each.
template <int K>
__device__ __forceinline__ void load_time_f32(const TimeMats* __restrict__ tm, float* sM) {
  constexpr int KK = K * K;
  for (int i = threadIdx.x; i < KK; i += blockDim.x) {
    const float q = (float)tm->Qb[i];
    sM[i] = q;
    sM[KK + i] = (float)tm->Ub[i];
    sM[2 * KK + i] = (float)tm->Eb[i];
    sM[3 * KK + i] = (float)tm->Wt[i];
    sM[4 * KK + (i % K) * K + i / K] = q;
  }
}
// complex64 right-hand side (M~^dagger Wt (f - M~ c))_U (+ yx) of one subvolume, by a CTA of NT threads or, WARP, by
// one warp: a thread holds a point's K coefficients in registers, so residual, weight and H c need no pass over
// shared memory between them and the index maps are paid once per point instead of once per coefficient.
// sC: c on U + 2, sZ: Wt r on U + 1, sV: dsum + V0 on U + 1; sRhs [npad] with zeros in the padding.
// Synchronised on return.  sM may still be on its way when the call begins (the first barrier covers it).
template <int K, bool WARP>
__device__ __forceinline__ void sweep_rhs(const LevelGeom& L, const FineOp& g, const SweepBox& B, int tid, int NT,
                                          int npad, const float* sM, float* sV, float2* sC, float2* sZ, float2* sRhs,
                                          const float2* f, const float2* yx, const float2* c) {
  constexpr int KK = K * K;
  auto sync = [] {
    if (WARP) __syncwarp();
    else __syncthreads();
  };
  const int nbc = B.ec[0] * B.ec[1] * B.ec[2], nbf = B.ef[0] * B.ef[1] * B.ef[2], npts = B.e[0] * B.e[1] * B.e[2];
  overlap_wait();   // c and f are read from here on
  for (int t = tid; t < nbc; t += NT) {
    int lx, ly, lz;
    SweepBox::coords(t, B.dc0, B.dc1, lx, ly, lz);
    const int gx = B.oc[0] + lx, gy = B.oc[1] + ly, gz = B.oc[2] + lz;
    const bool in = fine_in(g, gx, gy, gz);
    const float2* src = in ? c + (size_t)((gz * g.n[1] + gy) * g.n[0] + gx) * K : c;
    if constexpr (K % 2 == 0) {
#pragma unroll
      for (int m = 0; m < K; m += 2) cp_async16_zf(sC + t * K + m, src + m, in);
    } else {
#pragma unroll
      for (int m = 0; m < K; ++m) cp_async_elem_zf(sC + t * K + m, src + m, in);
    }
  }
  const float dsum = (float)g.dsum;
  const float xo = (float)(g.lax == 0 ? g.x0[0] : (g.lax == 1 ? g.x0[1] : g.x0[2]));
  const float xh = (float)(g.lax == 0 ? g.h[0] : (g.lax == 1 ? g.h[1] : g.h[2]));
  const float wx = -0.5f * (float)g.ih2[0], wy = -0.5f * (float)g.ih2[1], wz = -0.5f * (float)g.ih2[2];
  auto laser_x = [&](int gx, int gy, int gz) { return xo + (float)(g.lax == 0 ? gx : (g.lax == 1 ? gy : gz)) * xh; };
  // h = H v at a point of a staged field (records of K, strides dy, dz points)
  auto apply = [&](const float2* own, float dg, int dy, int dz, float2 (&v)[K], float2 (&h)[K]) {
    float2 a1[K], a2[K];
    rec_k<K>(own, v);
    rec_k<K>(own + K, a1);
    rec_k<K>(own - K, a2);
#pragma unroll
    for (int m = 0; m < K; ++m)
      h[m] = make_float2(dg * v[m].x + wx * (a1[m].x + a2[m].x), dg * v[m].y + wx * (a1[m].y + a2[m].y));
    if (L.dim > 1) {
      rec_k<K>(own + dy * K, a1);
      rec_k<K>(own - dy * K, a2);
#pragma unroll
      for (int m = 0; m < K; ++m) { h[m].x += wy * (a1[m].x + a2[m].x); h[m].y += wy * (a1[m].y + a2[m].y); }
    }
    if (L.dim > 2) {
      rec_k<K>(own + dz * K, a1);
      rec_k<K>(own - dz * K, a2);
#pragma unroll
      for (int m = 0; m < K; ++m) { h[m].x += wz * (a1[m].x + a2[m].x); h[m].y += wz * (a1[m].y + a2[m].y); }
    }
  };
  // q.v, u.h and e.v of one row of the matrices at offsets 0 (Q or Q^T), U, E
  auto row_products = [&](const float* sQ, int m, const float2 (&v)[K], const float2 (&h)[K], float2& qv, float2& uh,
                          float2& ev) {
    float q[K], u[K], ee[K];
    row_k<K>(sQ + m * K, q);
    row_k<K>(sM + KK + m * K, u);
    row_k<K>(sM + 2 * KK + m * K, ee);
    qv = uh = ev = make_float2(0.f, 0.f);
#pragma unroll
    for (int n = 0; n < K; ++n) {
      qv.x = fmaf(q[n], v[n].x, qv.x); qv.y = fmaf(q[n], v[n].y, qv.y);
      uh.x = fmaf(u[n], h[n].x, uh.x); uh.y = fmaf(u[n], h[n].y, uh.y);
      ev.x = fmaf(ee[n], v[n].x, ev.x); ev.y = fmaf(ee[n], v[n].y, ev.y);
    }
  };
  // r = f - M~ c and z = Wt r on the footprint, zero outside the grid
  bool staged = false;
  for (int i = tid; i < nbf || !staged; i += NT) {
    int lx = 0, ly = 0, lz = 0;
    SweepBox::coords(i < nbf ? i : 0, B.df0, B.df1, lx, ly, lz);
    const int gx = B.of_[0] + lx, gy = B.of_[1] + ly, gz = B.of_[2] + lz;
    const bool in = i < nbf && fine_in(g, gx, gy, gz);
    const size_t p = (size_t)((gz * g.n[1] + gy) * g.n[0] + gx);
    float2 r[K];
#pragma unroll
    for (int m = 0; m < K; ++m) r[m] = make_float2(0.f, 0.f);
    float dg = 0.f;
    if (in) {
      dg = dsum + (float)g.V0[p];
      if (f) rec_k<K>(f + p * K, r);
    }
    if (!staged) {
      cp_async_wait_all();
      sync();
      staged = true;
    }
    if (i >= nbf) break;
    sV[i] = dg;
    float2 z[K];
#pragma unroll
    for (int m = 0; m < K; ++m) z[m] = make_float2(0.f, 0.f);
    if (in) {
      const float2* own =
          sC + (((L.dim > 2 ? lz + 1 : lz) * B.ec[1] + (L.dim > 1 ? ly + 1 : ly)) * B.ec[0] + lx + 1) * K;
      float2 v[K], h[K];
      apply(own, dg, B.ec[0], B.ec[0] * B.ec[1], v, h);
      const float xl = laser_x(gx, gy, gz);
#pragma unroll
      for (int m = 0; m < K; ++m) {
        float2 q, u, ev;
        row_products(sM, m, v, h, q, u, ev);
        r[m].x -= -q.y - u.x - xl * ev.x;
        r[m].y -= q.x - u.y - xl * ev.y;
      }
#pragma unroll
      for (int m = 0; m < K; ++m) {
        float wm[K];
        row_k<K>(sM + 3 * KK + m * K, wm);
#pragma unroll
        for (int n = 0; n < K; ++n) { z[m].x = fmaf(wm[n], r[n].x, z[m].x); z[m].y = fmaf(wm[n], r[n].y, z[m].y); }
      }
    }
    if constexpr (K % 2 == 0) {
#pragma unroll
      for (int m = 0; m < K; m += 2)
        *reinterpret_cast<float4*>(sZ + i * K + m) = make_float4(z[m].x, z[m].y, z[m + 1].x, z[m + 1].y);
    } else {
#pragma unroll
      for (int m = 0; m < K; ++m) sZ[i * K + m] = z[m];
    }
  }
  sync();
  // rhs = M~^dagger z = -i Qb^T z - Ub H z - x Eb z on U; padding 0
  for (int t = npts * K + tid; t < npad; t += NT) sRhs[t] = make_float2(0.f, 0.f);
  for (int i = tid; i < npts; i += NT) {
    int lx, ly, lz;
    SweepBox::coords(i, B.du0, B.du1, lx, ly, lz);
    const int fi = ((L.dim > 2 ? lz + 1 : lz) * B.ef[1] + (L.dim > 1 ? ly + 1 : ly)) * B.ef[0] + lx + 1;
    const int gx = B.o[0] + lx, gy = B.o[1] + ly, gz = B.o[2] + lz;
    const float xl = laser_x(gx, gy, gz);
    float2 v[K], h[K];
    apply(sZ + fi * K, sV[fi], B.ef[0], B.ef[0] * B.ef[1], v, h);
    const size_t p = (size_t)((gz * g.n[1] + gy) * g.n[0] + gx);
#pragma unroll
    for (int m = 0; m < K; ++m) {
      float2 q, u, ev;
      row_products(sM + 4 * KK, m, v, h, q, u, ev);
      float2 out = make_float2(q.y - u.x - xl * ev.x, -q.x - u.y - xl * ev.y);
      if (yx) {   // additive right-hand side (adjoint relaxation of G z = y)
        const float2 yv = yx[p * K + m];
        out.x += yv.x;
        out.y += yv.y;
      }
      sRhs[i * K + m] = out;
    }
  }
  sync();
}
// c of unknown t of U plus delta, with c_U still in sC.
template <int K>
__device__ __forceinline__ void sweep_update(const LevelGeom& L, const FineOp& g, const SweepBox& B, int t, float2 d,
                                             const float2* sC, float2* c) {
  const int i = t / K, m = t - i * K;
  int lx, ly, lz;
  SweepBox::coords(i, B.du0, B.du1, lx, ly, lz);
  const float2 v = sC[(((L.dim > 2 ? lz + 2 : lz) * B.ec[1] + (L.dim > 1 ? ly + 2 : ly)) * B.ec[0] + lx + 2) * K + m];
  c[(size_t)(((B.o[2] + lz) * g.n[1] + (B.o[1] + ly)) * g.n[0] + (B.o[0] + lx)) * K + m] =
      make_float2(v.x + d.x, v.y + d.y);
}

// One complex64 subvolume of a colour with a superblock factor per CTA.
// One colour of 128^3, K = 4, 4x4x4 subvolumes (4096 of them): 236 us = 3.8 TB/s of in-band factor bytes read
// once (the backward pass finds them in L2), against 319 us with 128 threads and 16-row steps; 96^3: 105
// against 157 us.  Bound by the latency of a CTA's phases:
// four CTAs per SM with one piece in flight (64 registers) beat three with two (108 us at 96^3) and two with three
// (116 us); an L2 prefetch of the band at the start of the CTA costs 7 us.
template <int NPAD, int K>
__global__ void __launch_bounds__(kSuperThreads, K <= 4 ? 4 : 2)
k_sweep_super(LevelGeom L, FineOp g, const TimeMats* __restrict__ tm, const float2* f, const float2* yx, float2* c,
              const float2* __restrict__ factors, int colour, FastDiv dn0, FastDiv dn1) {
  extern __shared__ __align__(16) unsigned char smem[];
  overlap_trigger();
  const int tid = threadIdx.x;
  SweepBox B;
  const float2* F = factors + (size_t)B.init(L, colour, blockIdx.x, dn0, dn1) * L.fsize;
  const SuperSmem S = super_smem(L, K);
  float* sM = reinterpret_cast<float*>(smem);
  float2* sC = reinterpret_cast<float2*>(smem + S.c);
  float2* sRhs = reinterpret_cast<float2*>(smem + S.rhs);       // right-hand side
  float2* sXs = sRhs + NPAD;                                    // solution
  float2* sY = sXs + NPAD;                                      // scratch of the solves
  float2* sPr = sY + 2 * NPAD;
  load_time_f32<K>(tm, sM);
  sweep_rhs<K, false>(L, g, B, tid, kSuperThreads, NPAD, sM, reinterpret_cast<float*>(smem + S.v), sC,
                      reinterpret_cast<float2*>(smem + S.z), sRhs, f, yx, c);
  subvol_solve_super<NPAD>(F, L.band, sRhs, sY, sPr, sXs);
  for (int t = tid; t < B.e[0] * B.e[1] * B.e[2] * K; t += kSuperThreads) sweep_update<K>(L, g, B, t, sXs[t], sC, c);
}

// ------------------------------------------------------------------------ finest sweep, small subvolumes
// complex64 subvolumes of at most 32 unknowns, whose factor is stored as X = inv(L): one warp per subvolume,
// four per CTA, so nothing waits on a CTA barrier and the time matrices are converted once for four.  The warp
// loads X (at most twelve 16-byte loads per lane) before it forms the right-hand side and uses the same
// registers for y = X rhs and x = X^dagger y: lane (row l / 4 of each group of eight, quarter l % 4 of each block's
// columns), the sums folded across the lanes so that each ends with one unknown.
// One colour of 256^2, K = 4, 4x2 subvolumes (2048 of them): 10.1 us; 128 threads per subvolume with the same
// inverse took 19.4 us, a third of it conversions of the time matrices and barriers.
constexpr int kSmallSweepWarps = 4;
__host__ __device__ __forceinline__ SuperSmem small_smem(const LevelGeom& L, int K) {
  const int nbc = (L.sub[0] + 4) * (L.dim > 1 ? L.sub[1] + 4 : 1) * (L.dim > 2 ? L.sub[2] + 4 : 1);
  const int nbf = (L.sub[0] + 2) * (L.dim > 1 ? L.sub[1] + 2 : 1) * (L.dim > 2 ? L.sub[2] + 2 : 1);
  SuperSmem s;   // per warp, after the time matrices; total: one warp's bytes
  s.v = 0;
  s.c = (nbf * 4 + 15) & ~15;
  s.z = s.c + ((nbc * K * 8 + 15) & ~15);
  s.rhs = s.z + ((nbf * K * 8 + 15) & ~15);
  s.total = s.rhs + 2 * 32 * 8;   // rhs, y
  return s;
}
template <int NPAD, int K>
__global__ void __launch_bounds__(32 * kSmallSweepWarps)
k_sweep_small(LevelGeom L, FineOp g, const TimeMats* __restrict__ tm, const float2* f, const float2* yx, float2* c,
              const float2* __restrict__ factors, int colour, FastDiv dn0, FastDiv dn1, int count) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NB = NPAD / LA_BLK, NG = NPAD / 8;   // blocks per side; groups of eight rows
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, row = l >> 2, q = l & 3;
  const int j = blockIdx.x * kSmallSweepWarps + w;
  overlap_trigger();
  float* sM = reinterpret_cast<float*>(smem);
  load_time_f32<K>(tm, sM);
  __syncthreads();
  if (j >= count) return;
  SweepBox B;
  const float2* F = factors + (size_t)B.init(L, colour, j, dn0, dn1) * L.fsize;
  // X[8 G + row][16 J + 4 q + ..] of the blocks J <= G / 2
  float4 X[NG][NB][2];
#pragma unroll
  for (int G = 0; G < NG; ++G)
#pragma unroll
    for (int J = 0; J <= G / 2; ++J)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        X[G][J][u] = __ldg(reinterpret_cast<const float4*>(F + tri_index(G / 2, J) * 256 +
                                                           (8 * (G & 1) + row) * LA_BLK + 4 * q + 2 * u));
  const SuperSmem S = small_smem(L, K);
  unsigned char* base = smem + ((5 * K * K * 4 + 15) & ~15) + w * S.total;
  float2* sC = reinterpret_cast<float2*>(base + S.c);
  float2* sRhs = reinterpret_cast<float2*>(base + S.rhs);
  float2* sY = sRhs + 32;
  sweep_rhs<K, true>(L, g, B, l, 32, NPAD, sM, reinterpret_cast<float*>(base), sC, reinterpret_cast<float2*>(base + S.z),
                     sRhs, f, yx, c);
  const float2 zero = make_float2(0.f, 0.f);
  {
    float2 a[NG];
#pragma unroll
    for (int G = 0; G < NG; ++G) a[G] = zero;
#pragma unroll
    for (int J = 0; J < NB; ++J)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 v = *reinterpret_cast<const float4*>(sRhs + LA_BLK * J + 4 * q + 2 * u);
#pragma unroll
        for (int G = 2 * J; G < NG; ++G) {
          cfma(a[G], make_float2(X[G][J][u].x, X[G][J][u].y), make_float2(v.x, v.y));
          cfma(a[G], make_float2(X[G][J][u].z, X[G][J][u].w), make_float2(v.z, v.w));
        }
      }
    // over the four quarters: lane q ends with group 2 (q & 1) + (q / 2) (NPAD 16: group q & 1)
    float2 s = fold(a[0], a[NG / 2], l & 1, 1);
    if constexpr (NG > 2) s = fold(s, fold(a[1], a[3], l & 1, 1), l & 2, 2);
    else s = reduce_xor(s, 2);
    const int G = NG > 2 ? 2 * (q & 1) + (q >> 1) : (q & 1);
    if (NG > 2 || q < 2) sY[8 * G + row] = s;
  }
  __syncwarp();
  float2 x[NB][4];
#pragma unroll
  for (int J = 0; J < NB; ++J)
#pragma unroll
    for (int u = 0; u < 4; ++u) x[J][u] = zero;
#pragma unroll
  for (int G = 0; G < NG; ++G) {
    const float2 y = sY[8 * G + row];
#pragma unroll
    for (int J = 0; J <= G / 2; ++J)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        cfma_conj(x[J][2 * u], make_float2(X[G][J][u].x, X[G][J][u].y), y);
        cfma_conj(x[J][2 * u + 1], make_float2(X[G][J][u].z, X[G][J][u].w), y);
      }
  }
  // over the eight rows (lane bits 2, 3, 4): column 4 q + 2 bit 2 + bit 3 of block bit 4
  float2 s[NB];
#pragma unroll
  for (int J = 0; J < NB; ++J)
    s[J] = fold(fold(x[J][0], x[J][2], l & 4, 4), fold(x[J][1], x[J][3], l & 4, 4), l & 8, 8);
  float2 d;
  if constexpr (NB > 1) d = fold(s[0], s[1], l & 16, 16);
  else d = reduce_xor(s[0], 16);
  const int t = (NB > 1 ? (l >> 4) * LA_BLK : 0) + 4 * q + ((l & 4) ? 2 : 0) + ((l & 8) ? 1 : 0);
  if ((NB > 1 || l < 16) && t < B.e[0] * B.e[1] * B.e[2] * K) sweep_update<K>(L, g, B, t, d, sC, c);
}

// ======================================================================== Galerkin-level sweep
// rhs = (g - G e)_U with G = sum_kk' Sigma_kk' (x) Theta_kk' from the stored stencils.  The
// subvolume's stencils (|U| x 9 x box) and e on U + 2 are staged in shared memory with
// coalesced loads first, so the stencil sums run from shared memory with short dependency
// chains: (i, kk', n) tasks form u = Sigma_kk' e, then (i, m) tasks combine the nine pairs.
template <typename R>
struct CoarseSmem {
  typedef typename C2<R>::T CT;
  R* P; CT* E; R* Sg; CT* U; CT* Rhs; CT* Y; CT* T; CT* Red;
};
__host__ __device__ inline size_t coarse_sg_count(const LevelGeom& L) {
  const size_t nptsmax = (size_t)L.sub[0] * L.sub[1] * L.sub[2];
  return (nptsmax * LA_NPAIR * box5_count(L.dim) + 3) & ~(size_t)3;
}
__host__ __device__ inline size_t coarse_box_count(const LevelGeom& L) {
  const int sx = L.sub[0] + 4, sy = L.dim > 1 ? L.sub[1] + 4 : 1, sz = L.dim > 2 ? L.sub[2] + 4 : 1;
  return (size_t)sx * sy * sz;
}
template <typename R>
__device__ inline CoarseSmem<R> coarse_smem_layout(unsigned char* smem, const LevelGeom& L, int K, int npad) {
  typedef typename C2<R>::T CT;
  CoarseSmem<R> m;
  const size_t nptsmax = (size_t)L.sub[0] * L.sub[1] * L.sub[2];
  m.P = reinterpret_cast<R*>(smem);
  m.E = reinterpret_cast<CT*>(m.P + LA_NPAIR * LA_KMAX * LA_KMAX);
  m.Sg = reinterpret_cast<R*>(m.E + coarse_box_count(L) * K);
  m.U = reinterpret_cast<CT*>(m.Sg + coarse_sg_count(L));
  m.Rhs = m.U + nptsmax * LA_NPAIR * K;
  m.Y = m.Rhs + npad;
  m.T = m.Y + npad;
  m.Red = m.T + LA_BLK;
  return m;
}

// Multiply-shift index maps of one subvolume: item -> (point, time function), point -> (x, y, z) in U
// and in U + 2 (the level's divisors for a full subvolume, the CTA's own for a ragged one).
struct SubvolDiv {
  FastDiv K, c0, c1, u0, u1;
  __device__ SubvolDiv(const LevelGeom& L, const int e[3]) {
    const bool full = e[0] == L.sub[0] && e[1] == L.sub[1] && e[2] == L.sub[2];
    K = L.fd_K;
    c0 = full ? L.fd_c[0] : make_fastdiv(e[0] + 4);
    c1 = full ? L.fd_c[1] : make_fastdiv(L.dim > 1 ? e[1] + 4 : 1);
    u0 = full ? L.fd_u[0] : make_fastdiv(e[0]);
    u1 = full ? L.fd_u[1] : make_fastdiv(e[1]);
  }
  __device__ __forceinline__ void item(int t, int& i, int& m) const {
    i = fdiv(t, K);
    m = t - i * K.d;
  }
  __device__ __forceinline__ static void coords(int i, const FastDiv& d0, const FastDiv& d1, int& x, int& y,
                                                int& z) {
    const int r = fdiv(i, d0);
    x = i - r * d0.d;
    z = fdiv(r, d1);
    y = r - z * d1.d;
  }
};

// Fills S.Rhs[0..npad) with (g - G e) on the subvolume with origin o and extent e (0 in padding).
template <typename R>
__device__ inline void coarse_rhs(const LevelGeom& L, const R* __restrict__ sigma,
                                  const TimeMats* __restrict__ tm, const typename C2<R>::T* gvec,
                                  const typename C2<R>::T* ev, const int o[3], const int e[3], int npad,
                                  const CoarseSmem<R>& S) {
  typedef typename C2<R>::T CT;
  const int K = tm->K, KK = K * K;
  const int tid = threadIdx.x, nthr = blockDim.x;
  int ec[3], oc[3];
  for (int a = 0; a < 3; ++a) {
    const bool used = a < L.dim;
    ec[a] = used ? e[a] + 4 : 1;  oc[a] = used ? o[a] - 2 : o[a];
  }
  const int nbc = ec[0] * ec[1] * ec[2], npts = e[0] * e[1] * e[2];
  const int nbox = box5_count(L.dim);
  const SubvolDiv dv(L, e);
  for (int i = tid; i < LA_NPAIR * KK; i += nthr) S.P[i] = (R)tm->P[i / KK][i % KK];
  // the stencils of U's points and e on U + 2 (zero outside the grid) reach shared memory by cp.async, every copy
  // of a thread in flight at once instead of one dependent load per loop trip; e once its writers have finished
  const int per_pt = LA_NPAIR * nbox;
  for (int t = tid; t < npts * per_pt; t += nthr) {
    const int i = fdiv(t, L.fd_pair), w = t - i * per_pt;
    int lx, ly, lz;
    SubvolDiv::coords(i, dv.u0, dv.u1, lx, ly, lz);
    const int p = ((o[2] + lz) * L.n[1] + (o[1] + ly)) * L.n[0] + (o[0] + lx);
    cp_async_real(S.Sg + t, sigma + (size_t)p * per_pt + w);
  }
  overlap_wait();
  for (int t = tid; t < nbc * K; t += nthr) {
    int i, m;
    dv.item(t, i, m);
    int lx, ly, lz;
    SubvolDiv::coords(i, dv.c0, dv.c1, lx, ly, lz);
    const int gx = oc[0] + lx, gy = oc[1] + ly, gz = oc[2] + lz;
    const bool in = gx >= 0 && gy >= 0 && gz >= 0 && gx < L.n[0] && gy < L.n[1] && gz < L.n[2];
    cp_async_elem_zf(S.E + t, in ? ev + (size_t)((gz * L.n[1] + gy) * L.n[0] + gx) * K + m : ev, in);
  }
  cp_async_wait_all();
  __syncthreads();
  // u[i][kk][n] = sum_o Sigma_kk[p_i][o] e[p_i + o][n]
  const int ry = L.dim > 1 ? 2 : 0, rz = L.dim > 2 ? 2 : 0;
  for (int t = tid; t < npts * LA_NPAIR * K; t += nthr) {
    int ikk, n;
    dv.item(t, ikk, n);
    const int i = ikk / LA_NPAIR;
    int lx, ly, lz;
    SubvolDiv::coords(i, dv.u0, dv.u1, lx, ly, lz);
    const int cx = lx + 2, cy = L.dim > 1 ? ly + 2 : ly, cz = L.dim > 2 ? lz + 2 : lz;
    const R* sg = S.Sg + (size_t)ikk * nbox;
    R ur0 = 0, ui0 = 0, ur1 = 0, ui1 = 0;
    int q = 0;
    for (int oz = -rz; oz <= rz; ++oz)
      for (int oy = -ry; oy <= ry; ++oy) {
        const CT* ep = S.E + (size_t)(((cz + oz) * ec[1] + (cy + oy)) * ec[0] + (cx - 2)) * K + n;
#pragma unroll
        for (int ox = 0; ox < 5; ++ox, ++q) {
          const R sv = sg[q];
          const CT v = ep[ox * K];
          if (ox & 1) { ur1 = fma(sv, v.x, ur1); ui1 = fma(sv, v.y, ui1); }
          else { ur0 = fma(sv, v.x, ur0); ui0 = fma(sv, v.y, ui0); }
        }
      }
    S.U[t] = mkc<CT>(ur0 + ur1, ui0 + ui1);
  }
  __syncthreads();
  // rhs[i, m] = g - sum_kk phase_kk sum_n P_kk[m][n] u[i][kk][n]   (pairs in fixed order)
  for (int t = tid; t < npad; t += nthr) {
    CT out = mkc<CT>(0, 0);
    if (t < npts * K) {
      int i, m;
      dv.item(t, i, m);
      int lx, ly, lz;
      SubvolDiv::coords(i, dv.u0, dv.u1, lx, ly, lz);
      const int p = ((o[2] + lz) * L.n[1] + (o[1] + ly)) * L.n[0] + (o[0] + lx);
      out = gvec[(size_t)p * K + m];
#pragma unroll
      for (int kk = 0; kk < LA_NPAIR; ++kk) {
        const CT* u = S.U + ((size_t)i * LA_NPAIR + kk) * K;
        const R* pr = S.P + kk * KK + m * K;
        R vr = 0, vi = 0;
        for (int nn = 0; nn < K; ++nn) { vr = fma(pr[nn], u[nn].x, vr); vi = fma(pr[nn], u[nn].y, vi); }
        const int ph = theta_phase(kk);
        if (ph == 0) { out.x -= vr; out.y -= vi; }
        else if (ph == 1) { out.x += vi; out.y -= vr; }   // -(i v)
        else { out.x -= vi; out.y += vr; }                // -(-i v)
      }
    }
    S.Rhs[t] = out;
  }
  __syncthreads();
}

template <typename R, int NPAD>
__global__ void __launch_bounds__(kSweepThreads)
k_sweep_coarse(LevelGeom L, const R* __restrict__ sigma, const TimeMats* __restrict__ tm,
               const typename C2<R>::T* gvec, typename C2<R>::T* ev,
               const typename C2<R>::T* __restrict__ factors, int colour) {
  typedef typename C2<R>::T CT;
  extern __shared__ __align__(16) unsigned char smem[];
  overlap_trigger();
  const int K = tm->K;
  const int b = colour_subvol(L, colour, blockIdx.x);
  int o[3], e[3];
  subvol_box(L, b, o, e);
  const int npts = e[0] * e[1] * e[2];
  constexpr bool kInv = factor_is_inverse<R, NPAD>();
  MaybeInverse<R, NPAD, kInv> inv;
  if constexpr (kInv) inv.load(factors + (size_t)b * L.fsize);
  CoarseSmem<R> S = coarse_smem_layout<R>(smem, L, K, NPAD);
  coarse_rhs<R>(L, sigma, tm, gvec, ev, o, e, NPAD, S);
  if constexpr (kInv) {
    inv.solve(S.Rhs, S.Y, S.Red);
  } else {
    subvol_solve<CT, NPAD>(L, factors + (size_t)b * L.fsize, S.Rhs, S.Y, S.T);
    __syncthreads();
  }
  const SubvolDiv dv(L, e);
  for (int t = threadIdx.x; t < npts * K; t += kSweepThreads) {
    int i, m;
    dv.item(t, i, m);
    int lx, ly, lz;
    SubvolDiv::coords(i, dv.u0, dv.u1, lx, ly, lz);
    const size_t gi = (size_t)(((o[2] + lz) * L.n[1] + (o[1] + ly)) * L.n[0] + (o[0] + lx)) * K + m;
    CT v = ev[gi], d;
    if constexpr (kInv) d = inv.result(S.Red, t);
    else d = S.Rhs[t];
    v.x += d.x;
    v.y += d.y;
    ev[gi] = v;
  }
}

// s = g - G e on every point of a Galerkin level, one CTA per subvolume (all colours at once).
template <typename R>
__global__ void __launch_bounds__(kSweepThreads)
k_gresid_tiles(LevelGeom L, const R* __restrict__ sigma, const TimeMats* __restrict__ tm,
               const typename C2<R>::T* gvec, const typename C2<R>::T* ev, typename C2<R>::T* out, int npad) {
  typedef typename C2<R>::T CT;
  extern __shared__ __align__(16) unsigned char smem[];
  overlap_trigger();
  const int K = tm->K;
  int o[3], e[3];
  subvol_box(L, blockIdx.x, o, e);
  const int npts = e[0] * e[1] * e[2];
  CoarseSmem<R> S = coarse_smem_layout<R>(smem, L, K, npad);
  coarse_rhs<R>(L, sigma, tm, gvec, ev, o, e, npad, S);
  const SubvolDiv dv(L, e);
  for (int t = threadIdx.x; t < npts * K; t += kSweepThreads) {
    int i, m;
    dv.item(t, i, m);
    int lx, ly, lz;
    SubvolDiv::coords(i, dv.u0, dv.u1, lx, ly, lz);
    out[(size_t)(((o[2] + lz) * L.n[1] + (o[1] + ly)) * L.n[0] + (o[0] + lx)) * K + m] = S.Rhs[t];
  }
}

// ======================================================================== host dispatch
// Several matrices per CTA only on levels of at least 512 subvolumes; a level with fewer (a small
// grid such as the 1D workload's 8) runs one matrix per CTA, so that its few matrices are
// factorised side by side instead of one after another in a single CTA.  (Per context: the
// batched workload's grids of 512 and more subvolumes, running concurrently, keep the grouping.)
constexpr int kFactorMultiMin = 512;
inline int factor_grid_mpc(const LevelGeom& L, int mpc) {
  return (L.nsub >= kFactorMultiMin && !L.one_per_cta) ? mpc : 1;
}

inline size_t factor_smem(const LevelGeom& L, int nptsmax, size_t csize, int mpc_) {
  const size_t ntri = (size_t)L.npad * (L.npad + 1) / 2;
  const size_t npair = (size_t)nptsmax * (nptsmax + 1) / 2;
  const size_t mpc = (size_t)mpc_;
  return mpc * (csize * (ntri + L.npad) + (size_t)L.npad * (csize / 2)) +
         sizeof(double) * LA_NPAIR * LA_KMAX * LA_KMAX + mpc * factor_pair_bytes((int)npair, L.npad, csize) +
         sizeof(int) * (mpc * npair + 1);
}
// Factors with inverted diagonal superblocks (k_factor_band): complex64, more than 128 unknowns and a band of
// at most 8 blocks, the largest window k_factor_band keeps in registers.
template <typename R>
inline bool factor_is_super(const LevelGeom& L) {
  return sizeof(R) == 4 && L.npad > LA_NPAD_MAX && L.band <= 8;
}
inline size_t sweep_fine_smem(const LevelGeom& L, int K, size_t rsize, size_t csize) {
  const int sx = L.sub[0] + 4, sy = L.dim > 1 ? L.sub[1] + 4 : 1, sz = L.dim > 2 ? L.sub[2] + 4 : 1;
  const size_t nbc = (size_t)sx * sy * sz;
  const size_t nbf = (size_t)(L.sub[0] + 2) * (L.dim > 1 ? L.sub[1] + 2 : 1) * (L.dim > 2 ? L.sub[2] + 2 : 1);
  return rsize * (4 * LA_KMAX * LA_KMAX + 2 * ((nbf + 3) & ~(size_t)3)) +
         csize * (nbc * K + 2 * nbf * K + 2 * (size_t)L.npad + LA_BLK + 128);
}
inline size_t sweep_coarse_smem(const LevelGeom& L, int K, size_t rsize, size_t csize) {
  const size_t nptsmax = (size_t)L.sub[0] * L.sub[1] * L.sub[2];
  return rsize * (LA_NPAIR * LA_KMAX * LA_KMAX + coarse_sg_count(L)) +
         csize * (coarse_box_count(L) * K + nptsmax * LA_NPAIR * K + 2 * (size_t)L.npad + LA_BLK + 128);
}

template <typename R, int NPAD, int mpc>
cudaError_t launch_factor_blk_m(const LevelGeom& L, const FineOp* fine, const R* sigma, const TimeMats* tm,
                                typename C2<R>::T* factors, int* status, cudaStream_t s) {
  typedef typename C2<R>::T CT;
  const int nptsmax = L.sub[0] * L.sub[1] * L.sub[2];
  const size_t smem = mpc * (sizeof(CT) * ((size_t)LA_BLK * NPAD + (size_t)(NPAD / LA_BLK) * 256) + sizeof(R) * NPAD) +
                      sizeof(R) * (LA_NPAIR * LA_KMAX * LA_KMAX +
                                   mpc * ((size_t)nptsmax * nptsmax * (fine ? 2 : LA_NPAIR) + nptsmax));
  auto kern = k_factor_blk<R, NPAD, mpc>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  FineOp g = fine ? *fine : FineOp{};
  kern<<<(L.nsub + mpc - 1) / mpc, kFactorThreads, smem, s>>>(L, g, fine ? 1 : 0, nptsmax, sigma, tm, factors, status);
  return cudaGetLastError();
}

template <typename R, int NPAD>
cudaError_t launch_factor_blk_n(const LevelGeom& L, const FineOp* fine, const R* sigma, const TimeMats* tm,
                                typename C2<R>::T* factors, int* status, cudaStream_t s) {
  constexpr int mpc = factor_c64_mpc(NPAD);
  if (mpc > 1 && factor_grid_mpc(L, mpc) == 1)
    return launch_factor_blk_m<R, NPAD, 1>(L, fine, sigma, tm, factors, status, s);
  return launch_factor_blk_m<R, NPAD, mpc>(L, fine, sigma, tm, factors, status, s);
}

// Wide subvolumes (more than LA_NPAD_MAX unknowns) exist on the finest level only.
template <typename R, int NPAD>
cudaError_t launch_factor_wide_n(const LevelGeom& L, const FineOp* fine, const TimeMats* tm,
                                 typename C2<R>::T* factors, int* status, cudaStream_t s) {
  typedef typename C2<R>::T CT;
  if (!fine) return cudaErrorInvalidValue;
  const size_t smem = wide_factor_smem(NPAD, sizeof(CT), sizeof(R));
  auto kern = k_factor_wide<R, NPAD>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  kern<<<L.nsub, kFactorThreads, smem, s>>>(L, *fine, tm, factors, status);
  return cudaGetLastError();
}

template <typename R, int NPAD, int W>
cudaError_t launch_factor_band_n(const LevelGeom& L, const FineOp* fine, const TimeMats* tm,
                                 typename C2<R>::T* factors, int* status, cudaStream_t s) {
  if (!fine) return cudaErrorInvalidValue;
  constexpr size_t smem = band_factor_smem<R, W>();
  auto kern = k_factor_band<R, NPAD, W>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  kern<<<L.nsub, kBandThreads, smem, s>>>(L, *fine, tm, factors, status);
  return cudaGetLastError();
}

template <typename R, int NPAD, int mpc>
cudaError_t launch_factor_m(const LevelGeom& L, const FineOp* fine, const R* sigma, const TimeMats* tm,
                            typename C2<R>::T* factors, int* status, cudaStream_t s) {
  const int nptsmax = L.sub[0] * L.sub[1] * L.sub[2];
  const size_t smem = factor_smem(L, nptsmax, sizeof(typename C2<R>::T), mpc);
  auto kern = k_factor<R, NPAD, mpc>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  FineOp g = fine ? *fine : FineOp{};
  kern<<<(L.nsub + mpc - 1) / mpc, kFactorThreads, smem, s>>>(L, g, fine ? 1 : 0, nptsmax, sigma, tm, factors, status);
  return cudaGetLastError();
}
template <typename R, int NPAD>
cudaError_t launch_factor_n(const LevelGeom& L, const FineOp* fine, const R* sigma, const TimeMats* tm,
                            typename C2<R>::T* factors, int* status, cudaStream_t s) {
  constexpr int mpc = factor_mpc(NPAD);
  if (mpc > 1 && factor_grid_mpc(L, mpc) == 1)
    return launch_factor_m<R, NPAD, 1>(L, fine, sigma, tm, factors, status, s);
  return launch_factor_m<R, NPAD, mpc>(L, fine, sigma, tm, factors, status, s);
}
template <int NPAD, int K>
cudaError_t launch_sweep_super(const LevelGeom& L, const FineOp& g, const TimeMats* tm, const float2* f,
                               const float2* yx, float2* c, const float2* factors, int colour, int nblocks,
                               cudaStream_t s) {
  const int smem = super_smem(L, K).total;
  auto kern = k_sweep_super<NPAD, K>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  const FastDiv dn0 = make_fastdiv((L.nb[0] - (colour & 1) + 1) / 2),
                dn1 = make_fastdiv((L.nb[1] - ((colour >> 1) & 1) + 1) / 2);
  return launch_overlapped(L.overlap, kOverlapSweep, kern, nblocks, kSuperThreads, smem, s, L, g, tm, f, yx, c, factors,
                           colour, dn0, dn1);
}
template <int NPAD, int K>
cudaError_t launch_sweep_small(const LevelGeom& L, const FineOp& g, const TimeMats* tm, const float2* f,
                               const float2* yx, float2* c, const float2* factors, int colour, int nblocks,
                               cudaStream_t s) {
  const size_t smem = ((5 * K * K * 4 + 15) & ~15) + (size_t)kSmallSweepWarps * small_smem(L, K).total;
  auto kern = k_sweep_small<NPAD, K>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  const FastDiv dn0 = make_fastdiv((L.nb[0] - (colour & 1) + 1) / 2),
                dn1 = make_fastdiv((L.nb[1] - ((colour >> 1) & 1) + 1) / 2);
  return launch_overlapped(L.overlap, kOverlapMax, kern, (nblocks + kSmallSweepWarps - 1) / kSmallSweepWarps,
                           32 * kSmallSweepWarps, smem, s, L, g, tm, f, yx, c, factors, colour, dn0, dn1, nblocks);
}
template <typename R, int NPAD>
cudaError_t launch_sweep_fine_n(const LevelGeom& L, const FineOp& g, const TimeMats* tm, int K,
                                const typename C2<R>::T* f, const typename C2<R>::T* yx, typename C2<R>::T* c,
                                const typename C2<R>::T* factors, int colour, cudaStream_t s) {
  const int nblocks = colour_count(L, colour);
  if (nblocks == 0) return cudaSuccess;
  if constexpr (factor_is_inverse<R, NPAD>()) {
#define LA_SMALL(KK) case KK: return launch_sweep_small<NPAD, KK>(L, g, tm, f, yx, c, factors, colour, nblocks, s)
    switch (K) {
      LA_SMALL(1); LA_SMALL(2); LA_SMALL(3); LA_SMALL(4); LA_SMALL(5); LA_SMALL(6); LA_SMALL(7); LA_SMALL(8);
      default: return cudaErrorInvalidValue;
    }
#undef LA_SMALL
  } else {
  if constexpr (sizeof(R) == 4 && NPAD > LA_NPAD_MAX) {
    if (factor_is_super<R>(L)) {
#define LA_SUPER(KK) case KK: return launch_sweep_super<NPAD, KK>(L, g, tm, f, yx, c, factors, colour, nblocks, s)
      switch (K) {   // 64 points at most: more than 128 unknowns need K >= 3
        LA_SUPER(3); LA_SUPER(4); LA_SUPER(5); LA_SUPER(6); LA_SUPER(7); LA_SUPER(8);
        default: return cudaErrorInvalidValue;
      }
#undef LA_SUPER
    }
  }
  const size_t smem = sweep_fine_smem(L, K, sizeof(R), sizeof(typename C2<R>::T));
  auto kern = k_sweep_fine<R, NPAD>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  return launch_overlapped(L.overlap && sizeof(R) == 4, kOverlapSweep, kern, nblocks, kSweepThreads, smem, s, L, g, tm, f,
                           yx, c, factors, colour);
  }
}
template <typename R, int NPAD>
cudaError_t launch_sweep_coarse_n(const LevelGeom& L, const R* sigma, const TimeMats* tm, int K,
                                  const typename C2<R>::T* gvec, typename C2<R>::T* e,
                                  const typename C2<R>::T* factors, int colour, cudaStream_t s) {
  const int nblocks = colour_count(L, colour);
  if (nblocks == 0) return cudaSuccess;
  const size_t smem = sweep_coarse_smem(L, K, sizeof(R), sizeof(typename C2<R>::T));
  auto kern = k_sweep_coarse<R, NPAD>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  return launch_overlapped(L.overlap && sizeof(R) == 4, kOverlapMax, kern, nblocks, kSweepThreads, smem, s, L, sigma, tm,
                           gvec, e, factors, colour);
}

template <typename R>
cudaError_t launch_gresid_tiles_r(const LevelGeom& L, const R* sigma, const TimeMats* tm, int K,
                                  const typename C2<R>::T* gvec, const typename C2<R>::T* e, typename C2<R>::T* out,
                                  cudaStream_t s) {
  const size_t smem = sweep_coarse_smem(L, K, sizeof(R), sizeof(typename C2<R>::T));
  auto kern = k_gresid_tiles<R>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (err != cudaSuccess) return err;
    attr_set = true;
  }
  if (smem > 227 * 1024) return cudaErrorInvalidValue;
  return launch_overlapped(L.overlap && sizeof(R) == 4, kOverlapMax, kern, L.nsub, kSweepThreads, smem, s, L, sigma, tm,
                           gvec, e, out, L.npad);
}

// finest-level sweeps and factorisations also take the wide sizes
#define LA_NPAD_DISPATCH_WIDE(NPADV, CALL) \
  switch (NPADV) {                    \
    case 192: return CALL(192);       \
    case 256: return CALL(256);       \
    default: break;                   \
  }

#define LA_NPAD_DISPATCH(NPADV, CALL) \
  switch (NPADV) {                    \
    case 16: return CALL(16);         \
    case 32: return CALL(32);         \
    case 48: return CALL(48);         \
    case 64: return CALL(64);         \
    case 96: return CALL(96);         \
    case 128: return CALL(128);       \
    default: return cudaErrorInvalidValue; \
  }

}  // namespace la
