// complex64 factorisation of subvolumes of at most 32 unknowns (Galerkin levels and small finest-level
// subvolumes of the mixed path): the inverse X = inv(L) of the Cholesky factor, as 16 x 16 blocks.
#include "k_subvol.cuh"

namespace la {
namespace {

// Warps per CTA on levels of at least kSmallManyMin matrices, eight per SM; with fewer, or factor_group 1, one.  Four
// convert the time matrices once, one spreads better and ends its CTA sooner.  The line is flat: with one / four warps
// 900, 1225, 1600 and 3600 matrices take 24 / 26, 29 / 30, 30 / 32 and 57 / 55 us (2D 4x2 x 4), 26 / 26, 31 / 31,
// 32 / 31 and 60 / 55 us (2x2 x 8), 27 / 28, 33 / 35, 35 / 36 and 67 / 65 us (4x4 x 2).
constexpr int kSmallWarps = 4, kSmallManyMin = 8 * kSms;

// The entries of H and H^2 that only the spacings enter, w_a = 1 / (2 h_a^2): w_a, w_a^2 and 2 sum w_a^2 (a point's
// neighbours away from the walls) in FP64, and rounded once w_a, w_a^2 and 2 w_x w_y, 2 w_x w_z, 2 w_y w_z.
struct SpacingWeights {
  double w[3], w2[3], inner;
  float f[3], f2[3], fxy, fxz, fyz;
};
inline SpacingWeights spacing_weights(const FineOp& g) {
  SpacingWeights s;
  for (int a = 0; a < 3; ++a) {
    s.w[a] = 0.5 * g.ih2[a];
    s.w2[a] = s.w[a] * s.w[a];
    s.f[a] = (float)s.w[a];
    s.f2[a] = (float)s.w2[a];
  }
  s.inner = 2.0 * (s.w2[0] + s.w2[1] + s.w2[2]);
  s.fxy = (float)(2.0 * s.w[0] * s.w[1]);
  s.fxz = (float)(2.0 * s.w[0] * s.w[2]);
  s.fyz = (float)(2.0 * s.w[1] * s.w[2]);
  return s;
}

// NP lanes per matrix (one or two matrices per warp), lane r holding row r.  G_UU is assembled in registers
// and replaced in place by the inverse of its unit lower factor: G = L D L^dagger, step j subtracts
// (a_rj / d_j) u from the rows r > j, where u_c = conj(a_cj) for the columns c > j still to eliminate and u_c = row j
// of inv(L) for c < j, so that column j, once eliminated, holds inv(L)'s.  Rows are scaled by d^{-1/2} at the
// end.  The registers rotate by one column per step (register c holds column (j + c) mod NP), which keeps the
// loop rolled without a dynamic register index; u passes through shared memory, 16 bytes a load.
// H and H^2 of a finest-level point pair are formed in FP64 and rounded once (D_i + D_j may cancel), as the larger
// shared-memory factorisations do.  No barrier but the warp's: 7200 matrices of 32 unknowns (8 points x 4) take
// 96 us (the same with the pairs in FP32), half of the issue slots busy, against 161 us for four matrices per
// 256-thread CTA with two barriers per column.
template <int NP, int K, bool FINE>
__global__ void __launch_bounds__(32 * kSmallWarps)
k_factor_small(LevelGeom L, FineOp g, SpacingWeights sw, const float* __restrict__ sigma,
               const TimeMats* __restrict__ tm, float2* __restrict__ factors, int* __restrict__ status) {
  constexpr int KK = K * K, JMAX = NP / K;   // points of a full subvolume of this size class, at most
  __shared__ float sP[LA_NPAIR * KK], sPd[2 * KK];
  // FINE, per point: D = dsum + V0; the entries that D enters, rounded from FP64: H and H^2 on the diagonal, H^2 of the
  // links to the lower neighbours in the subvolume along x, y, z
  __shared__ double sD[kSmallWarps][FINE ? 32 : 1];
  __shared__ float sE[kSmallWarps][5][FINE ? 32 : 1], sX[kSmallWarps][32];
  // (H, H^2) of the point pairs i >= j, which K rows each look up: a table from K = 4 on, below that formed where they
  // are used (4000 matrices, K = 4 with 8 points: 59 us, 67 us without a table; 576, K = 3 with 8 points: 21.7 us,
  // 23.1 us with one; 4000, K = 1 with 32 points: 72 us, 86 us with a table of entries formed in FP64 pair by pair)
  constexpr bool kTable = FINE && K >= 4;
  constexpr int NPAIR = JMAX * (JMAX + 1) / 2;
  __shared__ float2 sHH[kSmallWarps][kTable ? (32 / NP) * NPAIR : 1];
  __shared__ int sXYZ[kSmallWarps][32];
  __shared__ __align__(16) float2 sBuf[kSmallWarps][2][32];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, r = lane & (NP - 1), half = lane / NP;
  const int b = (blockIdx.x * (blockDim.x >> 5) + w) * (32 / NP) + half;
  const bool real = b < L.nsub;   // lanes past the last subvolume work on an identity and store nothing
  for (int i = tid; i < LA_NPAIR * KK; i += blockDim.x) sP[i] = (float)tm->P[i / KK][i % KK];
  int o[3] = {0, 0, 0}, e[3] = {1, 1, 1}, npts = 0;
  if (real) {
    subvol_box(L, b, o, e);
    npts = e[0] * e[1] * e[2];
  }
  const int s0 = half * NP;
  if (r < npts) {
    int lx, ly, lz;
    local_coords(r, e, lx, ly, lz);
    sXYZ[w][s0 + r] = lx | (ly << 8) | (lz << 16);
    if (FINE) {
      const int px = o[0] + lx, py = o[1] + ly, pz = o[2] + lz;
      sD[w][s0 + r] = g.dsum + g.V0[(pz * g.n[1] + py) * g.n[0] + px];
      sX[w][s0 + r] = (float)fine_x(g, px, py, pz);
    }
  }
  __syncthreads();
  for (int i = tid; i < KK; i += blockDim.x) {
    sPd[i] = sP[KK + i] - sP[3 * KK + i];
    sPd[KK + i] = sP[2 * KK + i] - sP[6 * KK + i];
  }
  if (FINE && r < npts) {   // one point per lane: the FP64 pipe takes a warp's instruction 16 cycles, whoever is active
    const int x = sXYZ[w][s0 + r], l3[3] = {x & 255, (x >> 8) & 255, x >> 16}, below[3] = {1, e[0], e[0] * e[1]};
    const double D = sD[w][s0 + r];
    double d2 = fma(D, D, sw.inner);   // less w_a^2 for each neighbour beyond a Dirichlet wall; unused axes have w = 0
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int p = o[a] + l3[a];
      if (a < g.dim && p == 0) d2 -= sw.w2[a];
      if (a < g.dim && p + 1 == g.n[a]) d2 -= sw.w2[a];
      if (l3[a] > 0) sE[w][2 + a][s0 + r] = (float)(-sw.w[a] * (D + sD[w][s0 + r - below[a]]));
    }
    sE[w][0][s0 + r] = (float)D;
    sE[w][1][s0 + r] = (float)d2;
  }
  __syncthreads();
  // (H, H^2) of points i and j <= i, (dx, dy, dz) apart: in x-fastest order a neighbour j is i's lower one on its axis
  auto h_h2 = [&](int i, int dx, int dy, int dz) {
    const int ax = abs(dx), ay = abs(dy), az = abs(dz), a1 = ax + ay + az;
    if (a1 == 0) return make_float2(sE[w][0][s0 + i], sE[w][1][s0 + i]);
    if (a1 == 1) return make_float2(ax ? -sw.f[0] : (ay ? -sw.f[1] : -sw.f[2]), sE[w][ax ? 2 : (ay ? 3 : 4)][s0 + i]);
    float H2 = 0.f;
    if (a1 == 2) {
      H2 = ax ? (ay ? sw.fxy : sw.fxz) : sw.fyz;
      if (ax == 2) H2 = sw.f2[0];
      if (ay == 2) H2 = sw.f2[1];
      if (az == 2) H2 = sw.f2[2];
    }
    return make_float2(0.f, H2);
  };
  if constexpr (kTable) {
    for (int p = r; p < npts * (npts + 1) / 2; p += NP) {
      int a = (int)((sqrtf(8.f * (float)p + 1.f) - 1.f) * 0.5f);
      while (a * (a + 1) / 2 > p) --a;
      while ((a + 1) * (a + 2) / 2 <= p) ++a;
      const int xa = sXYZ[w][s0 + a], xq = sXYZ[w][s0 + p - a * (a + 1) / 2];
      sHH[w][half * NPAIR + p] =
          h_h2(a, (xq & 255) - (xa & 255), ((xq >> 8) & 255) - ((xa >> 8) & 255), (xq >> 16) - (xa >> 16));
    }
    __syncwarp();
  }
  // row r = (point i, time function m)
  const int i = r / K, m = r - i * K;
  const bool row_in = i < npts;
  float2 v[NP];
#pragma unroll
  for (int c = 0; c < NP; ++c) v[c] = make_float2(c == r ? 1.f : 0.f, 0.f);
  if (row_in) {
    const int xi = sXYZ[w][s0 + i];
    const int ix = xi & 255, iy = (xi >> 8) & 255, iz = xi >> 16;
    float Xi = 0.f;
    const float* sg = nullptr;
    const int nbox = box5_count(L.dim);
    if (FINE) {
      Xi = sX[w][s0 + i];
    } else {
      sg = sigma + sigma_offset(((o[2] + iz) * L.n[1] + (o[1] + iy)) * L.n[0] + (o[0] + ix), 0, 0, nbox);
    }
#pragma unroll
    for (int j = 0; j < JMAX; ++j) {
      if (j > i) break;   // lower triangle (the upper halves of the rows are never read)
      const int xj = sXYZ[w][s0 + j];
      const int dx = (xj & 255) - ix, dy = ((xj >> 8) & 255) - iy, dz = (xj >> 16) - iz;
      if (FINE) {
        const float2 hh = kTable ? sHH[w][kTable ? half * NPAIR + i * (i + 1) / 2 + j : 0] : h_h2(i, dx, dy, dz);
        const float H = hh.x, H2 = hh.y;
        const float Xj = sX[w][s0 + j];
#pragma unroll
        for (int n = 0; n < K; ++n) {
          const int mn = m * K + n;
          float re = H2 * sP[4 * KK + mn] + H * (Xj * sP[5 * KK + mn] + Xi * sP[7 * KK + mn]), im = H * sPd[mn];
          if (i == j) {
            re += sP[mn] + Xi * Xi * sP[8 * KK + mn];
            im += Xi * sPd[KK + mn];
          }
          v[j * K + n] = make_float2(re, im);
        }
      } else {
        const bool near = abs(dx) <= 2 && abs(dy) <= 2 && abs(dz) <= 2;
        const float* sj = sg + (near ? box5_index(L.dim, dx, dy, dz) : 0);
        float s9[LA_NPAIR];
#pragma unroll
        for (int kk = 0; kk < LA_NPAIR; ++kk) s9[kk] = near ? __ldg(sj + kk * nbox) : 0.f;
#pragma unroll
        for (int n = 0; n < K; ++n) {
          float re = 0.f, im = 0.f;
#pragma unroll
          for (int kk = 0; kk < LA_NPAIR; ++kk) {
            const float t = s9[kk] * sP[kk * KK + m * K + n];
            const int ph = theta_phase(kk);
            if (ph == 0) re += t; else if (ph == 1) im += t; else im -= t;
          }
          v[j * K + n] = make_float2(re, im);
        }
      }
    }
  }
  float scale = 1.f;
#pragma unroll 1
  for (int j = 0; j < NP; ++j) {
    const float2 a = v[0];
    float d = __shfl_sync(0xffffffffu, a.x, j, NP);
    if (!(d > 0.f)) {
      if (r == j) atomicOr(status, 1);
      d = 1.f;
    }
    if (r == j) scale = rsqrtf(d);
    const float rd = 1.f / d;
    const float2 gl = r > j ? make_float2(a.x * rd, a.y * rd) : make_float2(0.f, 0.f);
    float2* u = &sBuf[w][j & 1][s0];
    if (r == j) {
#pragma unroll
      for (int c = 0; c < NP; c += 2)
        *reinterpret_cast<float4*>(u + c) = make_float4(v[c].x, v[c].y, v[c + 1].x, v[c + 1].y);
    }
    __syncwarp();
    if (r > j) u[r - j] = make_float2(a.x, -a.y);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NP; c += 2) {
      const float4 q = *reinterpret_cast<const float4*>(u + c);
      if (c > 0) {
        v[c - 1].x = fmaf(-gl.x, q.x, fmaf(gl.y, q.y, v[c].x));
        v[c - 1].y = fmaf(-gl.x, q.y, fmaf(-gl.y, q.x, v[c].y));
      }
      v[c].x = fmaf(-gl.x, q.z, fmaf(gl.y, q.w, v[c + 1].x));
      v[c].y = fmaf(-gl.x, q.w, fmaf(-gl.y, q.z, v[c + 1].y));
    }
    v[NP - 1] = r > j ? make_float2(-gl.x, -gl.y) : make_float2(r == j ? 1.f : 0.f, 0.f);
  }
  if (!real) return;
  float2* F = factors + (size_t)b * L.fsize;
  const int br = r >> 4;
#pragma unroll
  for (int c = 0; c < NP; c += 2) {
    if ((c >> 4) > br) continue;
    *reinterpret_cast<float4*>(F + tri_index(br, c >> 4) * 256 + (r & 15) * LA_BLK + (c & 15)) =
        make_float4(scale * v[c].x, scale * v[c].y, scale * v[c + 1].x, scale * v[c + 1].y);
  }
}

template <int NP, int K>
cudaError_t launch_k(const LevelGeom& L, const FineOp* fine, const float* sigma, const TimeMats* tm, float2* factors,
                     int* status, cudaStream_t s) {
  const int warps = L.nsub >= kSmallManyMin && !L.one_per_cta ? kSmallWarps : 1, per = warps * (32 / NP);
  const int grid = (L.nsub + per - 1) / per;
  if (fine) {
    k_factor_small<NP, K, true><<<grid, 32 * warps, 0, s>>>(L, *fine, spacing_weights(*fine), sigma, tm, factors,
                                                            status);
  } else {
    k_factor_small<NP, K, false><<<grid, 32 * warps, 0, s>>>(L, FineOp{}, SpacingWeights{}, sigma, tm, factors, status);
  }
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_factor_small(const LevelGeom& L, const FineOp* fine, const float* sigma, const TimeMats* tm,
                                float2* factors, int* status, cudaStream_t s) {
#define LA_CALL(N, KK) case KK: return launch_k<N, KK>(L, fine, sigma, tm, factors, status, s)
#define LA_ALL(N) \
  switch (L.fd_K.d) { LA_CALL(N, 1); LA_CALL(N, 2); LA_CALL(N, 3); LA_CALL(N, 4); LA_CALL(N, 5); LA_CALL(N, 6); \
                      LA_CALL(N, 7); LA_CALL(N, 8); default: return cudaErrorInvalidValue; }
  if (L.npad == 16) LA_ALL(16)
  if (L.npad == 32) LA_ALL(32)
  return cudaErrorInvalidValue;
#undef LA_ALL
#undef LA_CALL
}

}  // namespace la
