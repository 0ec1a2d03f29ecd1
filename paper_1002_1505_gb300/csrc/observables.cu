// Incident field and scattering observables on the device.
//
// E_inc,j = e exp(i k . r_j) (guide, "Incident Polarization State"; plane wave
// along x_LF, expressed in the Target Frame), phase in FP64.
// Efficiency sums (Draine 1988, the formulas behind the guide's Q_ext, Q_abs,
// Q_pha), per RHS, FP64 accumulation, from the cached incident field:
//   S_ext = sum_j Im(E_j^* . P_j),  S_pha = sum_j Re(E_j^* . P_j),
//   S_abs = sum_j sum_a (-Im(alpha^{-1}_aa) - (2/3) k^3) |P_ja|^2
// (the host scales them by 4 pi k, 2 pi k and 4 pi k and divides by pi a_eff^2).
// Far field: F(n) = sum_j P_j exp(-i k n . r_j), from which the host forms
// f_ml = k^3 e_m . F (guide, eq. f_ml_def) and the Mueller matrix.
#include <algorithm>

#include "dda_internal.h"

namespace dda {

namespace {

constexpr int kT = 256;

template <typename C> __device__ __forceinline__ C mkc(double x, double y);
template <> __device__ __forceinline__ float2 mkc<float2>(double x, double y) { return make_float2((float)x, (float)y); }
template <> __device__ __forceinline__ double2 mkc<double2>(double x, double y) { return make_double2(x, y); }

template <typename C>
__global__ void k_einc(const int32_t* ijk, const double* org, const RhsGeom* rg, int64_t n, C* e) {
  const int b = blockIdx.y;
  const RhsGeom g = rg[b];
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double rx = ijk[3 * j] + org[0], ry = ijk[3 * j + 1] + org[1], rz = ijk[3 * j + 2] + org[2];
    const double ph = g.k[0] * rx + g.k[1] * ry + g.k[2] * rz;
    double sn, cs;
    sincos(ph, &sn, &cs);
    for (int c = 0; c < 3; ++c) {
      const double er = g.e[2 * c], ei = g.e[2 * c + 1];
      e[((int64_t)b * 3 + c) * n + j] = mkc<C>(er * cs - ei * sn, er * sn + ei * cs);
    }
  }
}

template <int NS>
__device__ __forceinline__ void bred(double (&v)[NS], double* out) {
  __shared__ double red[NS][kT / 32];
#pragma unroll
  for (int s = 0; s < NS; ++s)
    for (int o = 16; o > 0; o >>= 1) v[s] += __shfl_down_sync(0xffffffffu, v[s], o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int s = 0; s < NS; ++s) red[s][w] = v[s];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      double x = (threadIdx.x < (blockDim.x >> 5)) ? red[s][threadIdx.x] : 0.0;
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (threadIdx.x == 0) out[s] = x;
    }
  }
}

// efficiency sums from the cached incident field e [nrhs][3][N]
__global__ void k_qsum(const uint8_t* comp, const double2* __restrict__ e, const double2* ia, int ncomp, double kd,
                       const double2* p, int64_t n, double* part) {
  const int b = blockIdx.y;
  const double rr = (2.0 / 3.0) * kd * kd * kd;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    for (int c = 0; c < 3; ++c) {
      const int cc = comp ? comp[3 * j + c] : 0;  // composition of axis c
      const double2 ev = e[((int64_t)b * 3 + c) * n + j];
      const double2 pv = p[((int64_t)b * 3 + c) * n + j];
      // conj(E) * P
      const double re = ev.x * pv.x + ev.y * pv.y, im = ev.x * pv.y - ev.y * pv.x;
      acc[0] += im;
      acc[1] += re;
      const double2 a = ia[((int64_t)b * ncomp + cc) * 3 + c];
      acc[2] += (-a.y - rr) * (pv.x * pv.x + pv.y * pv.y);
    }
  }
  bred<3>(acc, part + ((int64_t)b * gridDim.x + blockIdx.x) * 4);
}

// the same sums for sites with a full symmetric alpha^{-1} (rotated dielectric frames):
// S_abs = sum_j { Im[P_j . (alpha_j^{-1})^* P_j^*] - (2/3) k^3 |P_j|^2 }
__global__ void k_qsum_t(const double2* __restrict__ e, const double2* __restrict__ iat, double kd,
                         const double2* __restrict__ p, int64_t n, double* part) {
  const int b = blockIdx.y;
  const double rr = (2.0 / 3.0) * kd * kd * kd;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    double2 P[3];
    for (int c = 0; c < 3; ++c) {
      const double2 ev = e[((int64_t)b * 3 + c) * n + j];
      const double2 pv = p[((int64_t)b * 3 + c) * n + j];
      P[c] = pv;
      acc[0] += ev.x * pv.y - ev.y * pv.x;
      acc[1] += ev.x * pv.x + ev.y * pv.y;
      acc[2] -= rr * (pv.x * pv.x + pv.y * pv.y);
    }
    const double2* m6 = iat + ((int64_t)b * n + j) * 6;
    for (int a = 0; a < 3; ++a)
      for (int c = 0; c < 3; ++c) {
        const int lo = a < c ? a : c, hi = a < c ? c : a;
        const double2 m = m6[lo == 0 ? hi : (lo == 1 ? 2 + hi : 5)];
        // Im[P_a conj(M_ac) conj(P_c)]
        const double2 t = make_double2(P[a].x * m.x + P[a].y * m.y, P[a].y * m.x - P[a].x * m.y);  // P_a conj(M)
        acc[2] += t.y * P[c].x - t.x * P[c].y;
      }
  }
  bred<3>(acc, part + ((int64_t)b * gridDim.x + blockIdx.x) * 4);
}

__global__ void k_qsum_fin(const double* part, int nblk, double* out3) {
  const int b = blockIdx.x;
  double v[3] = {0, 0, 0};
  for (int i = threadIdx.x; i < nblk; i += blockDim.x)
    for (int s = 0; s < 3; ++s) v[s] += part[((int64_t)b * nblk + i) * 4 + s];
  __shared__ double res[3];
  bred<3>(v, res);
  __syncthreads();
  if (threadIdx.x == 0)
    for (int s = 0; s < 3; ++s) out3[3 * b + s] = res[s];
}

// grid (nblk, ndir, nrhs): partial sums of P_j exp(-i k n.r_j) -> part[rhs][dir][blk][6], FP64.
// The phase factorises over the lattice axes, so each CTA first tabulates
// exp(-i k n_a (i + origin_a)) for its direction (box sum entries), then needs two
// complex products per site instead of a sine and cosine.
__global__ void k_far(const int32_t* ijk, const double* org, const double* nhat, double kd, const double2* p,
                      int ndir, int64_t n, int bx, int by, int bz, double* part) {
  extern __shared__ double2 ftab[];
  const int d = blockIdx.y, b = blockIdx.z;
  const double* nh = nhat + ((int64_t)b * ndir + d) * 3;
  const int nt = bx + by + bz;
  for (int i = threadIdx.x; i < nt; i += blockDim.x) {
    const int a = i < bx ? 0 : (i < bx + by ? 1 : 2);
    const int ii = a == 0 ? i : (a == 1 ? i - bx : i - bx - by);
    double sn, cs;
    sincos(-kd * nh[a] * ((double)ii + org[a]), &sn, &cs);
    ftab[i] = make_double2(cs, sn);
  }
  __syncthreads();
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double2 tx = ftab[ijk[3 * j]], ty = ftab[bx + ijk[3 * j + 1]], tz = ftab[bx + by + ijk[3 * j + 2]];
    const double2 txy = make_double2(tx.x * ty.x - tx.y * ty.y, tx.x * ty.y + tx.y * ty.x);
    const double cs = txy.x * tz.x - txy.y * tz.y, sn = txy.x * tz.y + txy.y * tz.x;
    for (int c = 0; c < 3; ++c) {
      const double2 pv = p[((int64_t)b * 3 + c) * n + j];
      acc[2 * c] += pv.x * cs - pv.y * sn;
      acc[2 * c + 1] += pv.x * sn + pv.y * cs;
    }
  }
  bred<6>(acc, part + (((int64_t)b * ndir + d) * gridDim.x + blockIdx.x) * 6);
}

// out[rhs][d0 + d] = the block partials of directions d0 .. d0 + nd - 1 in order; grid nrhs * nd
__global__ void k_far_fin(const double* part, int nblk, int nd, int ndir, int d0, double2* out) {
  const int64_t o = blockIdx.x, b = o / nd;  // rhs * nd + dir
  double v[6] = {0, 0, 0, 0, 0, 0};
  for (int i = threadIdx.x; i < nblk; i += blockDim.x)
    for (int s = 0; s < 6; ++s) v[s] += part[(o * nblk + i) * 6 + s];
  __shared__ double res[6];
  bred<6>(v, res);
  __syncthreads();
  if (threadIdx.x == 0)
    for (int c = 0; c < 3; ++c) out[(b * ndir + d0 + o - b * nd) * 3 + c] = make_double2(res[2 * c], res[2 * c + 1]);
}

// ------------------------------------------------------------------ many scattering directions
// The far-field phase of a lattice site factorises over the axes:
// exp(-i k n.r) = T_x[i] T_y[j] T_z[l] with T_a[i] = exp(-i k n_a (i + origin_a)); the tables
// are built in FP64 and stored in FP32, one set per (RHS, direction):
// tab[rd * nt + {0 | bx | bx + by} + i], nt = bx + by + bz.
__global__ void k_phase_tables(const double* __restrict__ nhat, int64_t nrd, const double* __restrict__ org, double kd,
                               int bx, int by, int bz, float2* __restrict__ tab) {
  const int nt = bx + by + bz;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nrd * nt; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t rd = t / nt;
    const int i = (int)(t - rd * nt);
    int a, ii;
    if (i < bx) { a = 0; ii = i; }
    else if (i < bx + by) { a = 1; ii = i - bx; }
    else { a = 2; ii = i - bx - by; }
    double sn, cs;
    sincos(-kd * nhat[rd * 3 + a] * ((double)ii + org[a]), &sn, &cs);
    tab[t] = make_float2((float)cs, (float)sn);
  }
}

// F[rhs][d] = sum_j P_j exp(-i k n_d . r_j) for kDirPerCta directions per CTA: grid (site blocks,
// direction chunks, nrhs); per-thread FP32 sums over its sites, then FP64 across the block.
constexpr int kDirPerCta = 8;
__global__ void __launch_bounds__(kT) k_far_many(const int32_t* __restrict__ ijk, const double2* __restrict__ p,
                                                 int64_t n, int ndir, int bx, int by, int bz,
                                                 const float2* __restrict__ tab, double* __restrict__ part) {
  extern __shared__ float2 stab[];
  const int nt = bx + by + bz;
  const int b = blockIdx.z, d0 = blockIdx.y * kDirPerCta;
  const int nd = min(kDirPerCta, ndir - d0);
  const float2* src = tab + ((int64_t)b * ndir + d0) * nt;
  for (int i = threadIdx.x; i < nd * nt; i += blockDim.x) stab[i] = src[i];
  __syncthreads();
  float acc[kDirPerCta][6];
#pragma unroll
  for (int dd = 0; dd < kDirPerCta; ++dd)
#pragma unroll
    for (int s = 0; s < 6; ++s) acc[dd][s] = 0.f;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const int ix = ijk[3 * j], iy = bx + ijk[3 * j + 1], iz = bx + by + ijk[3 * j + 2];
    float2 pv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 v = p[((int64_t)b * 3 + c) * n + j];
      pv[c] = make_float2((float)v.x, (float)v.y);
    }
#pragma unroll
    for (int dd = 0; dd < kDirPerCta; ++dd) {
      if (dd < nd) {
        const float2* t = stab + dd * nt;
        const float2 tx = t[ix], ty = t[iy], tz = t[iz];
        const float2 txy = make_float2(tx.x * ty.x - tx.y * ty.y, tx.x * ty.y + tx.y * ty.x);
        const float2 ph = make_float2(txy.x * tz.x - txy.y * tz.y, txy.x * tz.y + txy.y * tz.x);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          acc[dd][2 * c] = fmaf(pv[c].x, ph.x, fmaf(-pv[c].y, ph.y, acc[dd][2 * c]));
          acc[dd][2 * c + 1] = fmaf(pv[c].x, ph.y, fmaf(pv[c].y, ph.x, acc[dd][2 * c + 1]));
        }
      }
    }
  }
  double v[kDirPerCta * 6];
#pragma unroll
  for (int dd = 0; dd < kDirPerCta; ++dd)
#pragma unroll
    for (int s = 0; s < 6; ++s) v[dd * 6 + s] = (double)acc[dd][s];
  bred<kDirPerCta * 6>(v, part + (((int64_t)b * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * (kDirPerCta * 6));
}

// sum the site-block partials: out[rhs][d][3] (complex)
__global__ void k_far_many_fin(const double* __restrict__ part, int nblk, int nchunk, int ndir,
                               double2* __restrict__ out) {
  const int rc = blockIdx.x;  // rhs * nchunk + chunk
  const int b = rc / nchunk, ch = rc - b * nchunk;
  for (int s = threadIdx.x; s < kDirPerCta * 6; s += blockDim.x) {
    double v = 0.0;
    for (int i = 0; i < nblk; ++i) v += part[((int64_t)rc * nblk + i) * (kDirPerCta * 6) + s];
    const int d = ch * kDirPerCta + s / 6;
    if (d < ndir) {
      const int q = s % 6;
      double* o = reinterpret_cast<double*>(out + ((int64_t)b * ndir + d) * 3);
      o[q] = v;
    }
  }
}

// ------------------------------------------------------------------ far field by box rows
// The same sums organised by the box's x rows.  With c the row's centre and sites paired as
// x = c -+ delta, sum_x P e^{-ik n_x x} = e^{-ik n_x c} sum_u [P+ cos(phi_u) + i P- sin(phi_u)], where
// P+- = P(c + delta_u) +- P(c - delta_u) does not depend on the direction: four real products per
// pair, component and direction instead of eight, and the y, z and centre phases are applied once
// per row.  Tables per direction set (one per orientation; its nb polarizations share it):
// tab[set][i][ndp], direction fastest, i = u (cos, sin of phi_u), then y (with the centre phase),
// then z.  The work follows the box, so callers take it only for boxes that sites fill well
// (far_by_rows).
__device__ __forceinline__ double row_angle(const double* nh, const double* org, double kd, int nx, int i, int U,
                                            int ny) {
  const double c = 0.5 * (nx - 1);
  if (i < U) return -kd * nh[0] * (c - i);
  if (i < U + ny) return -kd * (nh[1] * ((double)(i - U) + org[1]) + nh[0] * (org[0] + c));
  return -kd * nh[2] * ((double)(i - U - ny) + org[2]);
}
// RUN consecutive entries of one section per thread.  T2 = float2: the first entry and the step by
// sincos, the others by FP64 products (error ~1e-15, far below the FP32 rounding of the entry);
// T2 = double2: sincos each.
constexpr int kRun = 16, kRun64 = 1;
template <typename T2, int RUN>
__global__ void k_row_tables(const double* __restrict__ nhat, int nb, int ndir, int ndp, const double* __restrict__ org,
                             double kd, int nx, int ny, int nz, T2* __restrict__ tab) {
  const int U = (nx + 1) / 2, nt = U + ny + nz;
  const int d = blockIdx.x * blockDim.x + threadIdx.x, set = blockIdx.z;
  if (d >= ndp) return;
  int s = blockIdx.y, i0, i1;  // section run
  const int ru = (U + RUN - 1) / RUN, ry = (ny + RUN - 1) / RUN;
  if (s < ru) { i0 = s * RUN; i1 = min(U, i0 + RUN); }
  else if (s < ru + ry) { i0 = U + (s - ru) * RUN; i1 = min(U + ny, i0 + RUN); }
  else { i0 = U + ny + (s - ru - ry) * RUN; i1 = min(nt, i0 + RUN); }
  const double* nh = nhat + ((int64_t)set * nb * ndir + min(d, ndir - 1)) * 3;
  T2* out = tab + (int64_t)set * nt * ndp + d;
  double sn, cs;
  const double a0 = row_angle(nh, org, kd, nx, i0, U, ny);
  sincos(a0, &sn, &cs);
  if constexpr (sizeof(T2) == sizeof(float2)) {
    double ws, wc;
    sincos(i1 > i0 + 1 ? row_angle(nh, org, kd, nx, i0 + 1, U, ny) - a0 : 0.0, &ws, &wc);
    for (int i = i0; i < i1; ++i) {
      out[(int64_t)i * ndp] = make_float2((float)cs, (float)sn);
      const double t = cs * wc - sn * ws;
      sn = cs * ws + sn * wc;
      cs = t;
    }
  } else {
    for (int i = i0; i < i1; ++i) {
      if (i > i0) sincos(row_angle(nh, org, kd, nx, i, U, ny), &sn, &cs);
      out[(int64_t)i * ndp] = make_double2(cs, sn);
    }
  }
}

// running FP32 sum carried as a pair (two-sum)
struct PairSum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(hi, v), z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v, z)));
    hi = t;
  }
};

// Many directions, FP32 products.  A thread owns two directions, a CTA 2 kRowT directions of one set
// and a run of rows, staged in shared memory as P+ and P- pairs that every thread reads by broadcast;
// a row's sum is FP32 (at most half the box's x length of terms), rows are added in pair sums.
// No one unit bounds it: issue 59 %, FMA 44 %, load write-back (the broadcasts) 46 % with 15 warps per SM.
// 131,072 sites x 2292 directions x 2 polarizations in 0.28 ms, where the site kernel took 7.66 ms (three
// table lookups and two complex products per site and direction, and 48 FP64 block sums per CTA at 1/64 of
// the FP32 rate).
// grid (nblk, ndp / (2 kRowT), nsets); part[set][blk][nb * 6][ndp].
constexpr int kRowT = 128;
template <int NB>
__global__ void __launch_bounds__(kRowT) k_far_rows(const int32_t* __restrict__ map, const double2* __restrict__ p,
                                                    int64_t n, int nx, int ny, int nz, int ndp,
                                                    const float2* __restrict__ tab, int rb, double* __restrict__ part) {
  extern __shared__ float4 srow[];  // [rb][U][NB * 3]: P+ (re, im), P- (re, im)
  constexpr int Q = NB * 3;
  const int U = (nx + 1) / 2, nt = U + ny + nz, nrows = ny * nz;
  int* occ = reinterpret_cast<int*>(srow + (size_t)rb * U * Q);
  const int set = blockIdx.z, d0 = blockIdx.y * 2 * kRowT + threadIdx.x;
  const int r_beg = (int)((int64_t)nrows * blockIdx.x / gridDim.x);
  const int r_end = (int)((int64_t)nrows * (blockIdx.x + 1) / gridDim.x);
  const float2* tx = tab + (int64_t)set * nt * ndp + d0;
  PairSum acc[2][2 * Q];
  for (int rb0 = r_beg; rb0 < r_end; rb0 += rb) {
    const int nr = min(rb, r_end - rb0);
    __syncthreads();
    for (int i = threadIdx.x; i < nr; i += kRowT) occ[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < nr * U; i += kRowT) {
      const int r = i / U, u = i - r * U;
      const int32_t* m = map + (int64_t)(rb0 + r) * nx;
      const int32_t ia = m[u], ib = (nx - 1 - u != u) ? m[nx - 1 - u] : -1;
      if (ia >= 0 || ib >= 0) occ[r] = 1;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const double2* pq = p + ((int64_t)set * Q + q) * n;
        const double2 a = ia >= 0 ? pq[ia] : make_double2(0.0, 0.0);
        const double2 b = ib >= 0 ? pq[ib] : make_double2(0.0, 0.0);
        const bool mid = nx - 1 - u == u;  // its own partner: sin(phi_u) = 0
        srow[(size_t)i * Q + q] = make_float4((float)(b.x + a.x), (float)(b.y + a.y), mid ? 0.f : (float)(b.x - a.x),
                                              mid ? 0.f : (float)(b.y - a.y));
      }
    }
    __syncthreads();
    for (int r = 0; r < nr; ++r) {
      if (!occ[r]) continue;
      float row[2][2 * Q];
#pragma unroll
      for (int q = 0; q < 2 * Q; ++q) row[0][q] = row[1][q] = 0.f;
      const float4* s = srow + (size_t)r * U * Q;
#pragma unroll 4
      for (int u = 0; u < U; ++u) {
        const float2 t0 = __ldg(tx + (int64_t)u * ndp), t1 = __ldg(tx + (int64_t)u * ndp + kRowT);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const float4 v = s[u * Q + q];
          row[0][2 * q] = fmaf(v.x, t0.x, fmaf(-v.w, t0.y, row[0][2 * q]));
          row[0][2 * q + 1] = fmaf(v.y, t0.x, fmaf(v.z, t0.y, row[0][2 * q + 1]));
          row[1][2 * q] = fmaf(v.x, t1.x, fmaf(-v.w, t1.y, row[1][2 * q]));
          row[1][2 * q + 1] = fmaf(v.y, t1.x, fmaf(v.z, t1.y, row[1][2 * q + 1]));
        }
      }
      const int iz = (rb0 + r) / ny, iy = (rb0 + r) - iz * ny;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2 a = __ldg(tx + (int64_t)(U + iy) * ndp + k * kRowT);
        const float2 b = __ldg(tx + (int64_t)(U + ny + iz) * ndp + k * kRowT);
        const float2 ph = make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          acc[k][2 * q].add(fmaf(row[k][2 * q], ph.x, -row[k][2 * q + 1] * ph.y));
          acc[k][2 * q + 1].add(fmaf(row[k][2 * q], ph.y, row[k][2 * q + 1] * ph.x));
        }
      }
    }
  }
  double* o = part + ((int64_t)set * gridDim.x + blockIdx.x) * (2 * Q) * ndp + d0;
#pragma unroll
  for (int q = 0; q < 2 * Q; ++q) {
    o[(int64_t)q * ndp] = (double)acc[0][q].hi + (double)acc[0][q].lo;
    o[(int64_t)q * ndp + kRowT] = (double)acc[1][q].hi + (double)acc[1][q].lo;
  }
}

// out[rhs][d][3] = the row blocks' partials in order; grid (ceil(ndir/256), nb * 6, nsets)
__global__ void k_far_rows_fin(const double* __restrict__ part, int nblk, int ndir, int ndp, int nb,
                               double2* __restrict__ out) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y, set = blockIdx.z;
  if (d >= ndir) return;
  double v = 0.0;
#pragma unroll 8
  for (int i = 0; i < nblk; ++i) v += part[(((int64_t)set * nblk + i) * (nb * 6) + q) * ndp + d];
  double* o = reinterpret_cast<double*>(out + (((int64_t)set * nb + q / 6) * ndir + d) * 3);
  o[q % 6] = v;
}

// Few directions, FP64 throughout: a thread owns a row (grid-strided) and kFarDirs directions, so the
// direction-independent P+- are formed once per kFarDirs directions; the CTA's totals leave in the
// layout of k_far's partials.  Bound by the FP64 pipe (12 products per pair and direction plus the
// P+- sums): 131,072 sites x 38 directions x 2 polarizations in 0.19 ms, k_far 0.59 ms (20 products
// per site and a table of sincos per CTA).  grid (row blocks, ceil(ndir / kFarDirs), nrhs).
constexpr int kFarDirs = 4;
constexpr int kFarT = 128;
__global__ void __launch_bounds__(kFarT) k_far_rows64(const int32_t* __restrict__ map, const double2* __restrict__ p,
                                                      int64_t n, int nx, int ny, int nz, int ndir, int nb,
                                                      const double2* __restrict__ tab, double* __restrict__ part) {
  extern __shared__ double2 sx[];  // [U][kFarDirs]
  __shared__ double red[kFarDirs * 6][kFarT + 1];
  const int U = (nx + 1) / 2, nt = U + ny + nz, nrows = ny * nz;
  const int d0 = blockIdx.y * kFarDirs, b = blockIdx.z;
  const double2* t = tab + (int64_t)(b / nb) * nt * ndir;
  for (int i = threadIdx.x; i < U * kFarDirs; i += kFarT)
    sx[i] = t[(int64_t)(i / kFarDirs) * ndir + min(d0 + i % kFarDirs, ndir - 1)];
  __syncthreads();
  double acc[kFarDirs][6];
#pragma unroll
  for (int k = 0; k < kFarDirs; ++k)
#pragma unroll
    for (int s = 0; s < 6; ++s) acc[k][s] = 0.0;
  const double2* pb = p + (int64_t)b * 3 * n;
  for (int r = blockIdx.x * kFarT + threadIdx.x; r < nrows; r += gridDim.x * kFarT) {
    const int32_t* m = map + (int64_t)r * nx;
    double row[kFarDirs][6];
#pragma unroll
    for (int k = 0; k < kFarDirs; ++k)
#pragma unroll
      for (int s = 0; s < 6; ++s) row[k][s] = 0.0;
    for (int u = 0; u < U; ++u) {
      const bool mid = nx - 1 - u == u;
      const int32_t ia = m[u], ib = mid ? -1 : m[nx - 1 - u];
      if (ia < 0 && ib < 0) continue;
      double2 sp[3], sm[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double2 a = ia >= 0 ? pb[c * n + ia] : make_double2(0.0, 0.0);
        const double2 e = ib >= 0 ? pb[c * n + ib] : make_double2(0.0, 0.0);
        sp[c] = make_double2(e.x + a.x, e.y + a.y);
        sm[c] = mid ? make_double2(0.0, 0.0) : make_double2(e.x - a.x, e.y - a.y);
      }
#pragma unroll
      for (int k = 0; k < kFarDirs; ++k) {
        const double2 w = sx[u * kFarDirs + k];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          row[k][2 * c] = fma(sp[c].x, w.x, fma(-sm[c].y, w.y, row[k][2 * c]));
          row[k][2 * c + 1] = fma(sp[c].y, w.x, fma(sm[c].x, w.y, row[k][2 * c + 1]));
        }
      }
    }
    const int iz = r / ny, iy = r - iz * ny;
#pragma unroll
    for (int k = 0; k < kFarDirs; ++k) {
      const int d = min(d0 + k, ndir - 1);
      const double2 a = t[(int64_t)(U + iy) * ndir + d], e = t[(int64_t)(U + ny + iz) * ndir + d];
      const double2 ph = make_double2(a.x * e.x - a.y * e.y, a.x * e.y + a.y * e.x);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[k][2 * c] += row[k][2 * c] * ph.x - row[k][2 * c + 1] * ph.y;
        acc[k][2 * c + 1] += row[k][2 * c] * ph.y + row[k][2 * c + 1] * ph.x;
      }
    }
  }
  // block totals: one column of `red` per thread, then four threads per value and a shuffle
#pragma unroll
  for (int k = 0; k < kFarDirs; ++k)
#pragma unroll
    for (int s = 0; s < 6; ++s) red[k * 6 + s][threadIdx.x] = acc[k][s];
  __syncthreads();
  if (threadIdx.x < kFarDirs * 24) {
    const int v = threadIdx.x / 4, q = threadIdx.x % 4;
    double s = 0.0;
    for (int i = 0; i < kFarT / 4; ++i) s += red[v][q + 4 * i];
    s += __shfl_down_sync(0xffffffffu, s, 2);
    s += __shfl_down_sync(0xffffffffu, s, 1);
    const int d = d0 + v / 6;
    if (q == 0 && d < ndir) part[(((int64_t)b * ndir + d) * gridDim.x + blockIdx.x) * 6 + v % 6] = s;
  }
}

// ------------------------------------------------------------------ radiative force and torque
// Far-field moments for the torque: per (RHS, direction) g = sum_j P_j exp(-i k n.r_j) (3 complex)
// and T[c][a] = sum_j (r_j - r_cm)_c P_ja exp(-i k n.r_j) (9 complex), from the same FP32 phase
// tables; grid (site blocks, direction pairs, nrhs); per-thread FP32 sums, FP64 across the block.
constexpr int kMomDir = 2;
constexpr int kMomVals = 24;  // 12 complex per direction
__global__ void __launch_bounds__(kT) k_far_moments(const int32_t* __restrict__ ijk, const double2* __restrict__ p,
                                                    int64_t n, int ndir, int bx, int by, int bz, float sx, float sy,
                                                    float sz, const float2* __restrict__ tab,
                                                    double* __restrict__ part) {
  extern __shared__ float2 stab[];
  const int nt = bx + by + bz;
  const int b = blockIdx.z, d0 = blockIdx.y * kMomDir;
  const int nd = min(kMomDir, ndir - d0);
  const float2* src = tab + ((int64_t)b * ndir + d0) * nt;
  for (int i = threadIdx.x; i < nd * nt; i += blockDim.x) stab[i] = src[i];
  __syncthreads();
  float acc[kMomDir][kMomVals];
#pragma unroll
  for (int dd = 0; dd < kMomDir; ++dd)
#pragma unroll
    for (int s = 0; s < kMomVals; ++s) acc[dd][s] = 0.f;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const int i0 = ijk[3 * j], i1 = ijk[3 * j + 1], i2 = ijk[3 * j + 2];
    const float rpos[3] = {(float)i0 + sx, (float)i1 + sy, (float)i2 + sz};
    float2 pv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double2 v = p[((int64_t)b * 3 + c) * n + j];
      pv[c] = make_float2((float)v.x, (float)v.y);
    }
#pragma unroll
    for (int dd = 0; dd < kMomDir; ++dd) {
      if (dd < nd) {
        const float2* t = stab + dd * nt;
        const float2 tx = t[i0], ty = t[bx + i1], tz = t[bx + by + i2];
        const float2 txy = make_float2(tx.x * ty.x - tx.y * ty.y, tx.x * ty.y + tx.y * ty.x);
        const float2 ph = make_float2(txy.x * tz.x - txy.y * tz.y, txy.x * tz.y + txy.y * tz.x);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float2 q = make_float2(pv[a].x * ph.x - pv[a].y * ph.y, pv[a].x * ph.y + pv[a].y * ph.x);
          acc[dd][2 * a] += q.x;
          acc[dd][2 * a + 1] += q.y;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            acc[dd][6 + 2 * (3 * c + a)] = fmaf(rpos[c], q.x, acc[dd][6 + 2 * (3 * c + a)]);
            acc[dd][6 + 2 * (3 * c + a) + 1] = fmaf(rpos[c], q.y, acc[dd][6 + 2 * (3 * c + a) + 1]);
          }
        }
      }
    }
  }
  double v[kMomDir * kMomVals];
#pragma unroll
  for (int dd = 0; dd < kMomDir; ++dd)
#pragma unroll
    for (int s = 0; s < kMomVals; ++s) v[dd * kMomVals + s] = (double)acc[dd][s];
  bred<kMomDir * kMomVals>(v, part + (((int64_t)b * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                                         (kMomDir * kMomVals));
}

// sum the site-block partials: out[rhs][d][12] (complex: g_x g_y g_z, then T row-major [c][a])
__global__ void k_far_moments_fin(const double* __restrict__ part, int nblk, int nchunk, int ndir,
                                  double2* __restrict__ out) {
  const int rc = blockIdx.x;  // rhs * nchunk + chunk
  const int b = rc / nchunk, ch = rc - b * nchunk;
  for (int s = threadIdx.x; s < kMomDir * kMomVals; s += blockDim.x) {
    double v = 0.0;
    for (int i = 0; i < nblk; ++i) v += part[((int64_t)rc * nblk + i) * (kMomDir * kMomVals) + s];
    const int d = ch * kMomDir + s / kMomVals;
    if (d < ndir) {
      double* o = reinterpret_cast<double*>(out + ((int64_t)b * ndir + d) * 12);
      o[s % kMomVals] = v;
    }
  }
}

// Incident-field part of the force and torque, per RHS (FP64): out7[b] =
// { sum_j Re(P_j x E_j^*) (3), sum_j (r_j - r_cm) Im(P_j . E_j^*) (3), sum_j Im(P_j . E_j^*) }.
__global__ void k_torque_ext(const int32_t* __restrict__ ijk, const double2* __restrict__ e,
                             const double2* __restrict__ p, int64_t n, double sx, double sy, double sz,
                             double* __restrict__ part) {
  const int b = blockIdx.y;
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    double2 P[3], E[3];
    for (int c = 0; c < 3; ++c) {
      P[c] = p[((int64_t)b * 3 + c) * n + j];
      E[c] = e[((int64_t)b * 3 + c) * n + j];
    }
    // P x E^*: component a = P_b E_c^* - P_c E_b^*, real part
    for (int a = 0; a < 3; ++a) {
      const int b1 = (a + 1) % 3, c1 = (a + 2) % 3;
      acc[a] += (P[b1].x * E[c1].x + P[b1].y * E[c1].y) - (P[c1].x * E[b1].x + P[c1].y * E[b1].y);
    }
    double im = 0.0;  // Im(P . E^*)
    for (int c = 0; c < 3; ++c) im += P[c].y * E[c].x - P[c].x * E[c].y;
    acc[3] += ((double)ijk[3 * j] + sx) * im;
    acc[4] += ((double)ijk[3 * j + 1] + sy) * im;
    acc[5] += ((double)ijk[3 * j + 2] + sz) * im;
    acc[6] += im;
  }
  bred<7>(acc, part + ((int64_t)b * gridDim.x + blockIdx.x) * 8);
}

__global__ void k_torque_ext_fin(const double* part, int nblk, double* out7) {
  const int b = blockIdx.x;
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int i = threadIdx.x; i < nblk; i += blockDim.x)
    for (int s = 0; s < 7; ++s) v[s] += part[((int64_t)b * nblk + i) * 8 + s];
  __shared__ double res[7];
  bred<7>(v, res);
  __syncthreads();
  if (threadIdx.x == 0)
    for (int s = 0; s < 7; ++s) out7[7 * b + s] = res[s];
}

// ------------------------------------------------------------------ fields in or near the target
// E and B at kNfPts points per CTA from every dipole (retarded point-dipole fields, FP64), the
// contribution of dipoles closer than one lattice spacing scaled by phi(R) = R^4 (5 - 4 R);
// grid (point chunks, nrhs); out[rhs][point][12] = E (re, im) x 3, then B.
constexpr int kNfPts = 4;

// E and B of the point dipole P (complex 3-vector) at separation (dx, dy, dz) from it, times the
// weight w (the near suppression, and for periodic targets the Bloch phase is in P and the cutoff in
// w), added to acc[0..5] (E) and acc[6..11] (B):
//   E = e^{ikR} { k^2 (n x p) x n / R + [3 n (n.p) - p] (1/R^3 - i k/R^2) },  B = e^{ikR} (n x p) (k^2/R + i k/R^2)
__device__ __forceinline__ void dipole_term(double dx, double dy, double dz, const double2 (&P)[3], double kd, double w,
                                            double* acc) {
  const double R2 = dx * dx + dy * dy + dz * dz;
  const double R = sqrt(R2), iR = 1.0 / R;
  const double nv[3] = {dx * iR, dy * iR, dz * iR};
  const double k2 = kd * kd;
  double sn, cs;
  sincos(kd * R, &sn, &cs);
  double2 nxp[3];
  for (int a = 0; a < 3; ++a) {
    const int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
    nxp[a] = make_double2(nv[a1] * P[a2].x - nv[a2] * P[a1].x, nv[a1] * P[a2].y - nv[a2] * P[a1].y);
  }
  const double2 ndp = make_double2(nv[0] * P[0].x + nv[1] * P[1].x + nv[2] * P[2].x,
                                   nv[0] * P[0].y + nv[1] * P[1].y + nv[2] * P[2].y);
  const double2 f = make_double2(iR * iR * iR, -kd * iR * iR);  // (1/R^3 - i k/R^2)
  const double2 ph = make_double2(cs * w, sn * w);
  const double2 gb = make_double2(k2 * iR, kd * iR * iR);
  for (int a = 0; a < 3; ++a) {
    const int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
    // ((n x p) x n)_a = (nxp)_{a1} n_{a2} - (nxp)_{a2} n_{a1}
    const double2 t1 = make_double2((nxp[a1].x * nv[a2] - nxp[a2].x * nv[a1]) * k2 * iR,
                                    (nxp[a1].y * nv[a2] - nxp[a2].y * nv[a1]) * k2 * iR);
    const double2 u = make_double2(3.0 * nv[a] * ndp.x - P[a].x, 3.0 * nv[a] * ndp.y - P[a].y);
    const double2 t2 = make_double2(u.x * f.x - u.y * f.y, u.x * f.y + u.y * f.x);
    const double2 e = make_double2(t1.x + t2.x, t1.y + t2.y);
    acc[2 * a] += e.x * ph.x - e.y * ph.y;
    acc[2 * a + 1] += e.x * ph.y + e.y * ph.x;
    const double2 bb = make_double2(nxp[a].x * gb.x - nxp[a].y * gb.y, nxp[a].x * gb.y + nxp[a].y * gb.x);
    acc[6 + 2 * a] += bb.x * ph.x - bb.y * ph.y;
    acc[6 + 2 * a + 1] += bb.x * ph.y + bb.y * ph.x;
  }
}

// near suppression of a dipole closer than one lattice spacing: (R/d)^4 (5 - 4 R/d)
__device__ __forceinline__ double near_suppression(double R) { return R < 1.0 ? R * R * R * R * (5.0 - 4.0 * R) : 1.0; }

__global__ void __launch_bounds__(kT) k_near_field(const int32_t* __restrict__ ijk, const double* __restrict__ org,
                                                   const double2* __restrict__ p, int64_t n,
                                                   const double* __restrict__ pts, int64_t npts, double kd,
                                                   double* __restrict__ out) {
  const int b = blockIdx.y;
  const int64_t q0 = (int64_t)blockIdx.x * kNfPts;
  double acc[kNfPts * 12];
#pragma unroll
  for (int i = 0; i < kNfPts * 12; ++i) acc[i] = 0.0;
  double xq[kNfPts][3];
#pragma unroll
  for (int q = 0; q < kNfPts; ++q)
    for (int a = 0; a < 3; ++a) xq[q][a] = (q0 + q < npts) ? pts[(q0 + q) * 3 + a] : 1e300;
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    const double r[3] = {ijk[3 * j] + org[0], ijk[3 * j + 1] + org[1], ijk[3 * j + 2] + org[2]};
    double2 P[3];
    for (int c = 0; c < 3; ++c) P[c] = p[((int64_t)b * 3 + c) * n + j];
#pragma unroll
    for (int q = 0; q < kNfPts; ++q) {
      if (q0 + q >= npts) continue;
      const double dx = xq[q][0] - r[0], dy = xq[q][1] - r[1], dz = xq[q][2] - r[2];
      const double R2 = dx * dx + dy * dy + dz * dz;
      if (R2 == 0.0) continue;
      dipole_term(dx, dy, dz, P, kd, near_suppression(sqrt(R2)), acc + q * 12);
    }
  }
  __shared__ double res[kNfPts * 12];
  bred<kNfPts * 12>(acc, res);
  __syncthreads();
  for (int i = threadIdx.x; i < kNfPts * 12; i += blockDim.x) {
    const int q = i / 12;
    if (q0 + q < npts) out[((int64_t)b * npts + q0 + q) * 12 + (i % 12)] = res[i];
  }
}

// Periodic targets: the replicas R = (0, m P_y, l P_z), |m| <= my, |l| <= mz, of every dipole, with
// moment P e^{i k.R} and weight exp[-(gamma k D)^4] on top of the near suppression, terms with
// (gamma k D)^4 > 40 dropped.  grid (nsplit, point chunks, nrhs): CTA s takes every nsplit-th
// block of the (dipole, replica) pairs; part[(b * nsplit + s) * npts + q][12] partial sums, added
// in a fixed order by k_nf_sum.
__global__ void __launch_bounds__(kT) k_near_field_pbc(const int32_t* __restrict__ ijk, const double* __restrict__ org,
                                                       const double2* __restrict__ p, int64_t n,
                                                       const double* __restrict__ pts, int64_t npts, double kd,
                                                       double ky, double kz, double py, double pz, double gamma, int my,
                                                       int mz, double* __restrict__ part) {
  const int s = blockIdx.x, nsplit = gridDim.x, b = blockIdx.z;
  const int64_t q0 = (int64_t)blockIdx.y * kNfPts;
  double acc[kNfPts * 12];
#pragma unroll
  for (int i = 0; i < kNfPts * 12; ++i) acc[i] = 0.0;
  double xq[kNfPts][3];
#pragma unroll
  for (int q = 0; q < kNfPts; ++q)
    for (int a = 0; a < 3; ++a) xq[q][a] = (q0 + q < npts) ? pts[(q0 + q) * 3 + a] : 1e300;
  const int64_t nrep = (int64_t)(2 * my + 1) * (2 * mz + 1);
  const int64_t pairs = n * nrep;
  const double gk = gamma * kd;
  for (int64_t idx = (int64_t)s * blockDim.x + threadIdx.x; idx < pairs; idx += (int64_t)nsplit * blockDim.x) {
    const int64_t j = idx % n, rep = idx / n;
    const int m = (int)(rep / (2 * mz + 1)) - my, l = (int)(rep % (2 * mz + 1)) - mz;
    const double Ry = m * py, Rz = l * pz;
    double sn, cs;
    sincos(ky * Ry + kz * Rz, &sn, &cs);
    const double r[3] = {ijk[3 * j] + org[0], ijk[3 * j + 1] + org[1] + Ry, ijk[3 * j + 2] + org[2] + Rz};
    double2 P[3];
    for (int c = 0; c < 3; ++c) {
      const double2 v = p[((int64_t)b * 3 + c) * n + j];
      P[c] = make_double2(v.x * cs - v.y * sn, v.x * sn + v.y * cs);
    }
#pragma unroll
    for (int q = 0; q < kNfPts; ++q) {
      if (q0 + q >= npts) continue;
      const double dx = xq[q][0] - r[0], dy = xq[q][1] - r[1], dz = xq[q][2] - r[2];
      const double R2 = dx * dx + dy * dy + dz * dz;
      if (R2 == 0.0) continue;
      const double R = sqrt(R2), t = gk * R, t4 = t * t * t * t;
      if (t4 > 40.0) continue;
      dipole_term(dx, dy, dz, P, kd, near_suppression(R) * exp(-t4), acc + q * 12);
    }
  }
  __shared__ double res[kNfPts * 12];
  bred<kNfPts * 12>(acc, res);
  __syncthreads();
  for (int i = threadIdx.x; i < kNfPts * 12; i += blockDim.x) {
    const int q = i / 12;
    if (q0 + q < npts) part[(((int64_t)b * nsplit + s) * npts + q0 + q) * 12 + (i % 12)] = res[i];
  }
}

// out[b][q][i] = sum over s (in order) of part[b][s][q][i]
__global__ void k_nf_sum(const double* __restrict__ part, int nsplit, int64_t npts, int nrhs, double* __restrict__ out) {
  const int64_t total = (int64_t)nrhs * npts * 12;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / (npts * 12), rem = i - b * npts * 12;
    double acc = 0.0;
    for (int s = 0; s < nsplit; ++s) acc += part[((b * nsplit + s) * npts) * 12 + rem];
    out[i] = acc;
  }
}

}  // namespace

Err near_field(const int32_t* ijk, const double* origin3, const double2* p, int nrhs, int64_t n, const double* pts,
               int64_t npts, double kd, double* out, cudaStream_t st) {
  const int64_t nchunk = (npts + kNfPts - 1) / kNfPts;
  if (nchunk > 2147483647LL) return Err::make(DDA_EINVAL, "too many field points");
  k_near_field<<<dim3((unsigned)nchunk, nrhs), kT, 0, st>>>(ijk, origin3, p, n, pts, npts, kd, out);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}

Err near_field_pbc(const int32_t* ijk, const double* origin3, const double2* p, int nrhs, int64_t n, const double* pts,
                   int64_t npts, double kd, const double k_tf[3], double py, double pz, double gamma, int my, int mz,
                   double* part, int nsplit, double* out, cudaStream_t st) {
  const int64_t nchunk = (npts + kNfPts - 1) / kNfPts;
  if (nchunk > 65535 || nrhs > 65535 || nsplit < 1) return Err::make(DDA_EINVAL, "too many field points");
  k_near_field_pbc<<<dim3((unsigned)nsplit, (unsigned)nchunk, (unsigned)nrhs), kT, 0, st>>>(
      ijk, origin3, p, n, pts, npts, kd, k_tf[1], k_tf[2], py, pz, gamma, my, mz, part);
  DDA_CU(cudaGetLastError());
  const int64_t total = (int64_t)nrhs * npts * 12;
  k_nf_sum<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((total + kT - 1) / kT, 1216)), kT, 0, st>>>(
      part, nsplit, npts, nrhs, out);
  DDA_CU(cudaGetLastError());
  add_launches(2);
  return Err::Ok();
}

Err farfield_moments(const int32_t* ijk, const double* origin3, const double* nhat, double kd, const double2* p,
                     int nrhs, int ndir, int64_t n, const int box[3], const double shift[3], float2* tab, double* part,
                     int nblk, double2* out, cudaStream_t st) {
  const int nt = box[0] + box[1] + box[2];
  const int64_t nrd = (int64_t)nrhs * ndir;
  const int tb = (int)std::min<int64_t>((nrd * nt + kT - 1) / kT, 152 * 32);
  k_phase_tables<<<tb, kT, 0, st>>>(nhat, nrd, origin3, kd, box[0], box[1], box[2], tab);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  const int nchunk = (ndir + kMomDir - 1) / kMomDir;
  const size_t sm = sizeof(float2) * (size_t)kMomDir * nt;
  if (sm > 48 * 1024) return Err::make(DDA_EUNSUPPORTED, "target box too long for the phase tables");
  k_far_moments<<<dim3(nblk, nchunk, nrhs), kT, sm, st>>>(ijk, p, n, ndir, box[0], box[1], box[2], (float)shift[0],
                                                          (float)shift[1], (float)shift[2], tab, part);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  k_far_moments_fin<<<nrhs * nchunk, 64, 0, st>>>(part, nblk, nchunk, ndir, out);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}

Err torque_ext_sums(const int32_t* ijk, const double2* einc, const double2* p, int nrhs, int64_t n,
                    const double shift[3], double* part, int nblk, double* out7, cudaStream_t st) {
  k_torque_ext<<<dim3(nblk, nrhs), kT, 0, st>>>(ijk, einc, p, n, shift[0], shift[1], shift[2], part);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  k_torque_ext_fin<<<nrhs, kT, 0, st>>>(part, nblk, out7);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}

// The row-wise sums follow the box, the site-wise ones the sites: rows are taken while the box has at
// most `most` positions per site.  Measured on a 48^3 box with a share f of its positions occupied,
// rows against sites: 2292 directions, two polarizations, f = 1: 0.43 / 6.3 ms, 0.52: 0.36 / 2.8,
// 0.27: 0.29 / 1.3 (the row time hardly falls with f, the site time is proportional, so they meet
// near 16 positions per site; the line is at 8); 38 directions in FP64, f = 1: 0.28 / 0.58 ms,
// 0.52: 0.27 / 0.35, 0.27: 0.27 / 0.22 (line at 2).  Rows longer than 700 would not fit the row
// kernels' shared memory.
constexpr int kRowsMost = 8, kRowsMost64 = 2;
static bool far_by_rows(int64_t n, const int box[3], int most) {
  return (int64_t)box[0] * box[1] * box[2] <= most * n && box[0] <= 700;
}

FarPlan far_many_plan(int64_t n, const int box[3], int nrhs, int iorth, int ndir) {
  FarPlan f;
  f.rows = far_by_rows(n, box, kRowsMost) && (iorth == 1 || iorth == 2);
  f.nb = f.rows ? iorth : 1;
  const int64_t nt = f.rows ? (int64_t)(box[0] + 1) / 2 + box[1] + box[2] : (int64_t)box[0] + box[1] + box[2];
  f.ndp = f.rows ? (ndir + 2 * kRowT - 1) / (2 * kRowT) * (2 * kRowT) : ndir;
  // direction sets per pass: phase tables under ~256 MB
  const int64_t sets = std::max<int64_t>(1, std::min<int64_t>(nrhs / f.nb, (256ll << 20) / (f.ndp * nt * 8)));
  f.per = (int)sets * f.nb;
  f.tab_bytes = sizeof(float2) * (size_t)(sets * f.ndp * nt);
  if (f.rows) {
    // one wave of four CTAs per SM (what 108 registers allow), at least eight rows each
    const int64_t tiles = (f.ndp / (2 * kRowT)) * sets;
    f.nblk = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)box[1] * box[2] + 7) / 8, 608 / tiles));
    f.part_doubles = (size_t)sets * f.nblk * f.nb * 6 * f.ndp;
  } else {
    f.nblk = (int)std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, 64));
    f.part_doubles = (size_t)f.per * ((ndir + kDirPerCta - 1) / kDirPerCta) * f.nblk * (kDirPerCta * 6);
  }
  return f;
}

Err farfield_many(const int32_t* ijk, const int32_t* map, const double* origin3, const double* nhat, double kd,
                  const double2* p, int nrhs, int ndir, int64_t n, const int box[3], const FarPlan& f, float2* tab,
                  double* part, double2* out, cudaStream_t st) {
  const int nt = box[0] + box[1] + box[2];
  if (sizeof(float2) * (size_t)kDirPerCta * nt > 48 * 1024)
    return Err::make(DDA_EUNSUPPORTED, "target box too long for the phase tables");
  if (f.rows) {
    const int nx = box[0], ny = box[1], nz = box[2], U = (nx + 1) / 2, sets = nrhs / f.nb;
    auto runs = [](int v) { return (v + kRun - 1) / kRun; };
    k_row_tables<float2, kRun><<<dim3((unsigned)((f.ndp + 127) / 128), runs(U) + runs(ny) + runs(nz), sets), 128, 0, st>>>(
        nhat, f.nb, ndir, (int)f.ndp, origin3, kd, nx, ny, nz, tab);
    DDA_CU(cudaGetLastError());
    // rows staged at a time: about 24 KB (one row of the longest box, 350 pairs, takes 33.6 KB)
    const size_t row_bytes = sizeof(float4) * (size_t)U * f.nb * 3;
    const int rb = (int)std::max<size_t>(1, std::min<size_t>(32, 24576 / row_bytes));
    const size_t sm = rb * row_bytes + sizeof(int) * rb;
    const dim3 grid(f.nblk, (unsigned)(f.ndp / (2 * kRowT)), sets);
    if (f.nb == 2) k_far_rows<2><<<grid, kRowT, sm, st>>>(map, p, n, nx, ny, nz, (int)f.ndp, tab, rb, part);
    else k_far_rows<1><<<grid, kRowT, sm, st>>>(map, p, n, nx, ny, nz, (int)f.ndp, tab, rb, part);
    DDA_CU(cudaGetLastError());
    k_far_rows_fin<<<dim3((ndir + 255) / 256, f.nb * 6, sets), 256, 0, st>>>(part, f.nblk, ndir, (int)f.ndp, f.nb, out);
    DDA_CU(cudaGetLastError());
    add_launches(3);
    return Err::Ok();
  }
  const int64_t nrd = (int64_t)nrhs * ndir;
  const int tb = (int)std::min<int64_t>((nrd * nt + kT - 1) / kT, 152 * 32);
  k_phase_tables<<<tb, kT, 0, st>>>(nhat, nrd, origin3, kd, box[0], box[1], box[2], tab);
  DDA_CU(cudaGetLastError());
  const int nchunk = (ndir + kDirPerCta - 1) / kDirPerCta;
  const size_t sm = sizeof(float2) * (size_t)kDirPerCta * nt;
  k_far_many<<<dim3(f.nblk, nchunk, nrhs), kT, sm, st>>>(ijk, p, n, ndir, box[0], box[1], box[2], tab, part);
  DDA_CU(cudaGetLastError());
  k_far_many_fin<<<nrhs * nchunk, 64, 0, st>>>(part, f.nblk, nchunk, ndir, out);
  DDA_CU(cudaGetLastError());
  add_launches(3);
  return Err::Ok();
}

template <typename C>
Err incident_field(const int32_t* ijk, const double* origin3, const RhsGeom* rg, int nrhs, int64_t n, C* e,
                   cudaStream_t st) {
  const int nb = (int)std::min<int64_t>((n + kT - 1) / kT, 1024);
  k_einc<C><<<dim3(nb, nrhs), kT, 0, st>>>(ijk, origin3, rg, n, e);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}
template Err incident_field<float2>(const int32_t*, const double*, const RhsGeom*, int, int64_t, float2*, cudaStream_t);
template Err incident_field<double2>(const int32_t*, const double*, const RhsGeom*, int, int64_t, double2*,
                                     cudaStream_t);

Err qsums(const uint8_t* comp, const double2* einc, const double2* ia, int ncomp, double kd, const double2* p,
          int nrhs, int64_t n, double* out3, RedBuf rb, cudaStream_t st) {
  k_qsum<<<dim3(rb.nblk, nrhs), kT, 0, st>>>(comp, einc, ia, ncomp, kd, p, n, rb.part);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  k_qsum_fin<<<nrhs, kT, 0, st>>>(rb.part, rb.nblk, out3);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}

Err qsums_tensor(const double2* einc, const double2* iat, double kd, const double2* p, int nrhs, int64_t n,
                 double* out3, RedBuf rb, cudaStream_t st) {
  k_qsum_t<<<dim3(rb.nblk, nrhs), kT, 0, st>>>(einc, iat, kd, p, n, rb.part);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  k_qsum_fin<<<nrhs, kT, 0, st>>>(rb.part, rb.nblk, out3);
  DDA_CU(cudaGetLastError());
  add_launches(1);
  return Err::Ok();
}

// row blocks of the row-wise far field
static int far_row_blocks(const int box[3]) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)box[1] * box[2] + kFarT - 1) / kFarT, 512));
}
static bool far_rows64(int nrhs, int64_t n, const int box[3]) { return far_by_rows(n, box, kRowsMost64) && nrhs <= 65535; }
// Its scratch for one direction: a column of the phase tables of each direction set, and the row blocks'
// partials of each RHS.  Directions beyond kFarScratch's worth take further passes, in whole direction
// groups: a pass of 64 MiB is thousands of CTAs, and with 32 RHS, 2000 directions and a 111 x 128 x 160 box
// the scratch of a single pass was 0.84 GB.
static size_t far_rows64_doubles(int nrhs, int iorth, const int box[3]) {
  return (size_t)2 * (nrhs / iorth) * ((box[0] + 1) / 2 + box[1] + box[2]) + (size_t)6 * nrhs * far_row_blocks(box);
}
constexpr size_t kFarScratch = (size_t)64 << 20;
static int far_rows64_dirs(int nrhs, int iorth, int ndir, const int box[3]) {
  const size_t fit = kFarScratch / sizeof(double) / far_rows64_doubles(nrhs, iorth, box);
  return (int)std::min<size_t>({(size_t)ndir, std::max<size_t>(1, fit / kFarDirs) * kFarDirs, (size_t)65535 * kFarDirs});
}
size_t farfield_scratch(int nrhs, int iorth, int ndir, int64_t n, const int box[3], int nblk) {
  if (!far_rows64(nrhs, n, box)) return (size_t)6 * nrhs * ndir * nblk;
  return far_rows64_doubles(nrhs, iorth, box) * far_rows64_dirs(nrhs, iorth, ndir, box);
}

Err farfield(const int32_t* ijk, const int32_t* map, const double* origin3, const double* nhat, double kd,
             const double2* p, int nrhs, int iorth, int ndir, int64_t n, const int box[3], double2* out,
             double* scratch, int nblk, cudaStream_t st) {
  const size_t sm = sizeof(double2) * (size_t)(box[0] + box[1] + box[2]);
  if (sm > 48 * 1024) return Err::make(DDA_EUNSUPPORTED, "target box too long for the far-field phase tables");
  if (far_rows64(nrhs, n, box)) {
    const int nx = box[0], ny = box[1], nz = box[2], U = (nx + 1) / 2, sets = nrhs / iorth;
    const int nrb = far_row_blocks(box), per = far_rows64_dirs(nrhs, iorth, ndir, box);
    auto runs = [](int v) { return (v + kRun64 - 1) / kRun64; };
    for (int d0 = 0; d0 < ndir; d0 += per) {
      const int nd = std::min(per, ndir - d0);
      double2* tab = reinterpret_cast<double2*>(scratch);
      double* part = scratch + 2 * (size_t)sets * nd * (U + ny + nz);
      k_row_tables<double2, kRun64><<<dim3((unsigned)((nd + 31) / 32), runs(U) + runs(ny) + runs(nz), sets), 32, 0, st>>>(
          nhat + (size_t)3 * d0, iorth, ndir, nd, origin3, kd, nx, ny, nz, tab);
      DDA_CU(cudaGetLastError());
      k_far_rows64<<<dim3(nrb, (nd + kFarDirs - 1) / kFarDirs, nrhs), kFarT, sizeof(double2) * U * kFarDirs, st>>>(
          map, p, n, nx, ny, nz, nd, iorth, tab, part);
      DDA_CU(cudaGetLastError());
      k_far_fin<<<(unsigned)(nrhs * (int64_t)nd), kT, 0, st>>>(part, nrb, nd, ndir, d0, out);
      DDA_CU(cudaGetLastError());
      add_launches(3);
    }
    return Err::Ok();
  }
  k_far<<<dim3(nblk, ndir, nrhs), kT, sm, st>>>(ijk, origin3, nhat, kd, p, ndir, n, box[0], box[1], box[2], scratch);
  DDA_CU(cudaGetLastError());
  k_far_fin<<<nrhs * ndir, kT, 0, st>>>(scratch, nblk, ndir, ndir, 0, out);
  DDA_CU(cudaGetLastError());
  add_launches(2);
  return Err::Ok();
}

}  // namespace dda
