// Bistatic RCS of a marched current envelope at chosen frequencies (Sec. 2.4): the
// frequency-domain currents of the march for a unit incident field, and their
// co-polarised far field.
//
//  * envelope convention x(t) = Re{x~(t) e^{j w_c t}}: the spectrum at f > 0 is half the
//    envelope's at Omega = 2 pi (f - f_c), and the half cancels between scattered and
//    incident fields;
//  * the current envelope is the CPPIF interpolant of its samples (Eq. 3), so
//    X~(Omega) = dt That(Omega dt) sum_l I_l e^{-j Omega l dt}, That(w) = int T(u) e^{-j w u} du;
//  * the incident envelope of Eq. 1 at the origin, g(t - t_d) e^{-j w_c t_d}, has the
//    transform E~(Omega) = sigma sqrt(2 pi) exp(-sigma^2 Omega^2 / 2) exp(-j (w_c + Omega) t_d);
//  * X~ / E~ is the frequency-domain current for the unit plane wave p e^{-j k k.r} at f
//    (the time-differentiated EFIE of Eq. 4 at one frequency is the frequency-domain
//    EFIE times j w), whose far field is E = -j w mu/(4 pi) e^{-j k r}/r F with
//    F = (I - r r) . sum_k I_k int S_k(r') e^{+j k r.r'} dS' (7-point cubature), and
//    sigma = 4 pi |pol . E r|^2.
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "aim_internal.h"
#include "rcs.h"
#include "setup_host.h"

namespace {

constexpr int kT = 256;

// acc[f][b][k] += w_f x[b][k] for the step's phases w_f = e^{-j Omega_f l dt}
__global__ void __launch_bounds__(kT) k_dft_accum(RcsPhases ph, long long n, const double2* __restrict__ x,
                                                   double2* __restrict__ acc) {
  for (long long i = blockIdx.x * (long long)kT + threadIdx.x; i < n; i += (long long)gridDim.x * kT) {
    const double2 v = x[i];
    for (int f = 0; f < ph.n; ++f) {
      const double2 w = ph.w[f];
      double2& a = acc[(size_t)f * n + i];
      a.x += w.x * v.x - w.y * v.y;
      a.y += w.x * v.y + w.y * v.x;
    }
  }
}

__global__ void __launch_bounds__(kT) k_scale_freq(RcsPhases s, long long n, double2* __restrict__ acc) {
  for (long long i = blockIdx.x * (long long)kT + threadIdx.x; i < n; i += (long long)gridDim.x * kT)
    for (int f = 0; f < s.n; ++f) {
      const double2 w = s.w[f];
      double2& a = acc[(size_t)f * n + i];
      a = make_double2(w.x * a.x - w.y * a.y, w.x * a.y + w.y * a.x);
    }
}

// The far field in three steps.  On a face the current is affine,
//   J(r) = sum_e c_e I_e (r - v_e) = a (r - C) - b,  c_e = sign l_e / (2 A), C the centroid,
// so a face carries one complex scalar and one complex vector per right-hand side
// (k_rcs_faces), whatever the direction.  For a direction the projected current at a
// cubature point is u . J = a u . (r - C) - u . b, u = pol - r (r . pol), and the sums over the
// 7 points  X = sum_q w_q u . (r_q - C) e^{jkr.r_q},  Y = sum_q w_q e^{jkr.r_q}  do not depend on
// the right-hand side (k_rcs_dirs); the points are the centroid and, for two fractions s,
// centroid + s (vertex - centroid), so their phases differ from the centroid's by small
// angles, which need the Taylor series of sine and cosine instead of a range reduction.
// The 7 points share the rounding of the centroid's phase, which does not average out over
// them as 7 separately rounded phases would: the centroid is held as an unevaluated sum of two
// doubles and its phase k r . C likewise (k_rcs_geom, k_rcs_dirs), the second part applied as
// a rotation to first order.  (Largest error over 40 directions of a 1920-RWG sphere at
// 300 MHz, of the largest value: 3.6-4.0e-16 with every point evaluated by itself, 7.9-8.9e-16
// with the rounded phase, 2.8-3.8e-16 with the two parts.)
// The kernels are bound by FP64 arithmetic: about 280 operations per face, direction and
// frequency plus 20 per right-hand side (each
// point evaluated by itself for every right-hand side took about 120 per point: 12.5 ms for
// 5120 faces, 288 directions, 3 frequencies and 2 waves, 2.3 ms now).
constexpr int kRcsB = 4;  // right-hand sides per pass
constexpr int kDirW = 2;  // warps per block of k_rcs_dirs

// a + b = result + err (the intrinsics keep a product before it from being contracted into it)
__device__ __forceinline__ double two_sum(double a, double b, double& err) {
  const double s = __dadd_rn(a, b), t = __dsub_rn(s, a);
  err = __dadd_rn(__dsub_rn(a, __dsub_rn(s, t)), __dsub_rn(b, t));
  return s;
}

// geo[12][nt]: the centroid C as a sum of two doubles per component, and two of the three
// vertices relative to it (they add up to zero)
__global__ void __launch_bounds__(kT) k_rcs_geom(int nt, const int* __restrict__ F, const double* __restrict__ V,
                                                 double* __restrict__ geo) {
  const int t = blockIdx.x * kT + threadIdx.x;
  if (t >= nt) return;
  for (int d = 0; d < 3; ++d) {
    const double v0 = V[3 * F[3 * t] + d], v1 = V[3 * F[3 * t + 1] + d], v2 = V[3 * F[3 * t + 2] + d];
    double e1, e2;
    const double s = two_sum(two_sum(v0, v1, e1), v2, e2), c = s / 3.0;
    const double lo = (fma(-3.0, c, s) + (e1 + e2)) / 3.0;
    geo[(size_t)d * nt + t] = c;
    geo[(size_t)(3 + d) * nt + t] = lo;
    geo[(size_t)(6 + d) * nt + t] = (v0 - c) - lo;
    geo[(size_t)(9 + d) * nt + t] = (v1 - c) - lo;
  }
}

// fc[fb][4][nt]: a, b_x, b_y, b_z of every face for right-hand sides b0 .. b0 + gridDim.y - 1 of
// frequencies f0 .. (fb = (f - f0) sb + (b - b0))
__global__ void __launch_bounds__(kT) k_rcs_faces(int nt, const double* __restrict__ geo,
                                                  const int* __restrict__ tbk, const double* __restrict__ tbs,
                                                  const int* __restrict__ tbf, const double* __restrict__ len,
                                                  const double* __restrict__ area, const double* __restrict__ V, int ns,
                                                  int nb, int b0, int sb, const double2* __restrict__ spec,
                                                  double2* __restrict__ fc) {
  const int t = blockIdx.x * kT + threadIdx.x, bs = blockIdx.y, f = blockIdx.z;
  if (t >= nt) return;
  double2 m[4] = {};
  if (b0 + bs < nb) {
    const double2* I = spec + ((size_t)f * nb + b0 + bs) * ns;
    for (int e = 0; e < 3; ++e) {
      const int k = tbk[3 * t + e];
      if (k < 0) continue;
      const double c = tbs[3 * t + e] * len[k] / (2.0 * area[t]);
      const double2 x = make_double2(c * I[k].x, c * I[k].y);
      const double* vf = V + 3 * tbf[3 * t + e];
      m[0].x += x.x;
      m[0].y += x.y;
      for (int d = 0; d < 3; ++d) {
        const double r = (vf[d] - geo[(size_t)d * nt + t]) - geo[(size_t)(3 + d) * nt + t];
        m[1 + d].x += x.x * r;
        m[1 + d].y += x.y * r;
      }
    }
  }
  for (int i = 0; i < 4; ++i) fc[((size_t)(f * sb + bs) * 4 + i) * nt + t] = m[i];
}

// sin and cos of |x| <= 1/2: Taylor series to x^15 and x^14 (remainders below 1e-18)
__device__ __forceinline__ void small_sincos(double x, double& s, double& c) {
  const double y = x * x;
  double p = -1.0 / 1307674368000.0, q = -1.0 / 87178291200.0;
  p = p * y + 1.0 / 6227020800.0;
  p = p * y - 1.0 / 39916800.0;
  p = p * y + 1.0 / 362880.0;
  p = p * y - 1.0 / 5040.0;
  p = p * y + 1.0 / 120.0;
  p = p * y - 1.0 / 6.0;
  s = x + x * (y * p);
  q = q * y + 1.0 / 479001600.0;
  q = q * y - 1.0 / 3628800.0;
  q = q * y + 1.0 / 40320.0;
  q = q * y - 1.0 / 720.0;
  q = q * y + 1.0 / 24.0;
  q = q * y - 0.5;
  c = 1.0 + y * q;
}

// part[fb][d][unit] = sum over the faces of a unit of u . int J e^{jkr.r'} dS'; a unit is 32 m
// consecutive faces, m to a lane, summed by one warp, and the units are a matter of the mesh
// alone: a value rounds the same whatever else is in the call.  Grid (nd, blocks, frequencies),
// a block's warps taking units blockIdx.y kDirW + warp, then gridDim.y kDirW further on.
// dirs: [nd][6] (rhat, pol); fk: [n_freq][2] (k, prefactor).
__global__ void __launch_bounds__(32 * kDirW) k_rcs_dirs(int nt, const double* __restrict__ geo,
                                                         const double* __restrict__ area,
                                                         const double2* __restrict__ fc, const double* __restrict__ fk,
                                                         const double* __restrict__ dirs, int nbc, int sb, int units,
                                                         int m, double2* __restrict__ part) {
  const int d = blockIdx.x, f = blockIdx.z, nd = gridDim.x, lane = threadIdx.x & 31;
  const double* rd = dirs + 6 * d;
  const double k = fk[2 * f];
  const double rp = rd[0] * rd[3] + rd[1] * rd[4] + rd[2] * rd[5];
  const double u[3] = {rd[3] - rd[0] * rp, rd[4] - rd[1] * rp, rd[5] - rd[2] * rp};
  // the orbits (p, p, 1 - 2p) of the rule: fraction 1 - 3p towards the vertex, and weights
  const double s15 = 3.8729833462074168852;  // sqrt 15
  const double fr[2] = {1.0 - (6.0 - s15) / 7.0, 1.0 - (6.0 + s15) / 7.0};
  const double w[2] = {(155.0 - s15) / 1200.0, (155.0 + s15) / 1200.0}, w0 = 9.0 / 40.0;
  for (int q = blockIdx.y * kDirW + (threadIdx.x >> 5); q < units; q += gridDim.y * kDirW) {
    const int end = min(nt, (q + 1) * 32 * m);
    double2 acc[kRcsB] = {};
    for (int t = q * 32 * m + lane; t < end; t += 32) {
      double v[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) v[i] = geo[(size_t)i * nt + t];
      // the vertices relative to the centroid, along the direction and the polarisation
      double ph[3], g[3];
      for (int i = 0; i < 2; ++i) {
        ph[i] = rd[0] * v[6 + 3 * i] + rd[1] * v[7 + 3 * i] + rd[2] * v[8 + 3 * i];
        g[i] = u[0] * v[6 + 3 * i] + u[1] * v[7 + 3 * i] + u[2] * v[8 + 3 * i];
      }
      ph[2] = -(ph[0] + ph[1]);
      g[2] = -(g[0] + g[1]);
      for (int i = 0; i < 3; ++i) ph[i] *= k;
      // the centroid's phase, pc + pl
      const double p0 = __dmul_rn(rd[0], v[0]), p1 = __dmul_rn(rd[1], v[1]), p2 = __dmul_rn(rd[2], v[2]);
      double t1, t2;
      const double ps = two_sum(two_sum(p0, p1, t1), p2, t2), pc = __dmul_rn(k, ps);
      const double pe = (fma(rd[0], v[0], -p0) + fma(rd[1], v[1], -p1) + fma(rd[2], v[2], -p2)) + (t1 + t2) +
                        (rd[0] * v[3] + rd[1] * v[4] + rd[2] * v[5]);
      const double pl = fma(k, pe, fma(k, ps, -pc));
      const double big = fmax(fabs(ph[0]), fmax(fabs(ph[1]), fabs(ph[2])));
      double2 X = make_double2(0.0, 0.0), Y = make_double2(w0, 0.0);
      for (int o = 0; o < 2; ++o) {
        double2 x = make_double2(0, 0), y = make_double2(0, 0);
        for (int i = 0; i < 3; ++i) {
          double sn, cs;
          if (big * fabs(fr[1]) <= 0.5 && big * fabs(fr[0]) <= 0.5) small_sincos(fr[o] * ph[i], sn, cs);
          else sincos(fr[o] * ph[i], &sn, &cs);
          y.x += cs;
          y.y += sn;
          x.x += g[i] * cs;
          x.y += g[i] * sn;
        }
        X.x += w[o] * fr[o] * x.x;
        X.y += w[o] * fr[o] * x.y;
        Y.x += w[o] * y.x;
        Y.y += w[o] * y.y;
      }
      double sn, cs;
      sincos(pc, &sn, &cs);
      const double A = area[t], c0 = cs;
      cs = A * fma(-pl, sn, cs);
      sn = A * fma(pl, c0, sn);
      X = make_double2(X.x * cs - X.y * sn, X.x * sn + X.y * cs);
      Y = make_double2(Y.x * cs - Y.y * sn, Y.x * sn + Y.y * cs);
#pragma unroll
      for (int b = 0; b < kRcsB; ++b)
        if (b < nbc) {
          const double2* c = fc + (size_t)(f * sb + b) * 4 * nt + t;
          const double2 a = c[0], bx = c[nt], by = c[2 * (size_t)nt], bz = c[3 * (size_t)nt];
          const double qx = u[0] * bx.x + u[1] * by.x + u[2] * bz.x, qy = u[0] * bx.y + u[1] * by.y + u[2] * bz.y;
          acc[b].x += a.x * X.x - a.y * X.y - (qx * Y.x - qy * Y.y);
          acc[b].y += a.x * X.y + a.y * X.x - (qx * Y.y + qy * Y.x);
        }
    }
    for (int b = 0; b < nbc; ++b) {
      const double2 s = warp_sum_c(acc[b]);
      if (lane == 0) part[((size_t)(f * sb + b) * nd + d) * units + q] = s;
    }
  }
}

// sig[f][b0 + bs][d], nd of the nd_all directions, = prefactor |sum of the units|^2, a warp per value
__global__ void __launch_bounds__(kT) k_rcs_finish(int nd, int nd_all, int units, int nb, int b0, int sb,
                                                   const double* __restrict__ fk, const double2* __restrict__ part,
                                                   double* __restrict__ sig) {
  const int d = blockIdx.x * (kT / 32) + (threadIdx.x >> 5), bs = blockIdx.y, f = blockIdx.z, lane = threadIdx.x & 31;
  if (d >= nd) return;
  const double2* p = part + ((size_t)(f * sb + bs) * nd + d) * units;
  double2 s = make_double2(0, 0);
  for (int q = lane; q < units; q += 32) {
    s.x += p[q].x;
    s.y += p[q].y;
  }
  s = warp_sum_c(s);
  if (lane == 0) sig[((size_t)f * nb + b0 + bs) * nd_all + d] = fk[2 * f + 1] * (s.x * s.x + s.y * s.y);
}

int blocks_for(long long n) { return (int)std::min<long long>((n + kT - 1) / kT, 152LL * 16); }

}  // namespace

std::complex<double> basis_spectrum(const TBasis& tb, double w) {
  std::vector<double> x, wt;
  host_gauss_legendre(24, x, wt);
  std::complex<double> s = 0.0;
  if (tb.kind == AIM_BLIF) {  // smooth on (-M, M): 24 points on each unit interval
    for (int j = -tb.Q; j < tb.Q; ++j)
      for (size_t i = 0; i < x.size(); ++i) {
        const double u = j + 0.5 + 0.5 * x[i];
        s += 0.5 * wt[i] * host_blif_value(tb, u) * std::exp(std::complex<double>(0.0, -w * u));
      }
    return s;
  }
  for (int j = 0; j <= tb.Q; ++j) {  // CPPIF piece (j-1, j]
    for (size_t i = 0; i < x.size(); ++i) {
      const double u = j - 0.5 + 0.5 * x[i];
      double T = 0;
      for (int p = tb.Q; p >= 0; --p) T = T * u + tb.coef[j][p];
      s += 0.5 * wt[i] * T * std::exp(std::complex<double>(0.0, -w * u));
    }
  }
  return s;
}

void rcs_dft_accum(aim_ctx* c, int nb, int l, int n_freq, const double* omega, const double2* x, double2* acc) {
  RcsPhases ph{};
  ph.n = n_freq;
  for (int f = 0; f < n_freq; ++f) {
    const double a = -omega[f] * l * c->dt;
    ph.w[f] = make_double2(std::cos(a), std::sin(a));
  }
  const long long n = (long long)nb * c->ns;
  k_dft_accum<<<blocks_for(n), kT, 0, c->stream>>>(ph, n, x, acc);
  AIM_CHECK_LAUNCH();
}

void rcs_scale(aim_ctx* c, int nb, const RcsPhases& s, double2* acc) {
  const long long n = (long long)nb * c->ns;
  k_scale_freq<<<blocks_for(n), kT, 0, c->stream>>>(s, n, acc);
  AIM_CHECK_LAUNCH();
}

// Faces per lane of a unit, of the mesh alone: 2, one on meshes of less than 16 blocks, more
// beyond 2048.  (One face per lane everywhere: the sums over lanes cost 4 % of the work; four:
// one direction of the 7680-RWG sphere takes 84 us instead of 53.)
static int rcs_m(const aim_ctx* c) {
  const int block = 32 * kDirW;
  return std::max(c->nt >= 16 * block ? 2 : 1, (c->nt + 2048 * block - 1) / (2048 * block));
}

void rcs_tables(aim_ctx* c) {
  c->d_geo = (double*)aim_alloc(c, (size_t)12 * c->nt * sizeof(double));
  k_rcs_geom<<<(c->nt + kT - 1) / kT, kT, 0, c->stream>>>(c->nt, c->d_tri, c->d_v, c->d_geo);
  AIM_CHECK_LAUNCH();
}

// Frequencies and directions of a pass: at most 64 MB of face currents and 64 MB of partial sums
// (at least one of each), for as many right-hand sides as a pass takes.
RcsPlan rcs_plan(const aim_ctx* c, int n_freq, int nb, int nd) {
  constexpr size_t kCap = (size_t(64) << 20) / sizeof(double2);
  RcsPlan p;
  p.nb = std::min(nb, kRcsB);
  p.units = (c->nt + 32 * rcs_m(c) - 1) / (32 * rcs_m(c));
  const size_t per_f = (size_t)p.nb * 4 * c->nt;
  p.nf = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_freq, kCap / per_f));
  p.nd = (int)std::max<size_t>(1, std::min<size_t>((size_t)nd, kCap / ((size_t)p.nf * p.nb * p.units)));
  p.faces = per_f * p.nf;
  p.elems = p.faces + (size_t)p.nf * p.nb * p.nd * p.units;
  return p;
}

void rcs_farfield(aim_ctx* c, const RcsPlan& p, int n_freq, int nb, const double2* spec, int nd, const double* dirs,
                  const double* fk, double2* work, double* sig) {
  double2* part = work + p.faces;
  const double* geo = c->d_geo;
  const int tb = (c->nt + kT - 1) / kT;
  for (int f0 = 0; f0 < n_freq; f0 += p.nf)
    for (int b0 = 0; b0 < nb; b0 += p.nb) {
      const int nf = std::min(p.nf, n_freq - f0), nbc = std::min(p.nb, nb - b0);
      k_rcs_faces<<<dim3(tb, nbc, nf), kT, 0, c->stream>>>(
          c->nt, geo, c->d_tbk, c->d_tbs, c->d_tbf, c->d_len, c->d_area, c->d_v, c->ns, nb, b0, p.nb,
          spec + (size_t)f0 * nb * c->ns, work);
      AIM_CHECK_LAUNCH();
      for (int d0 = 0; d0 < nd; d0 += p.nd) {
        const int n = std::min(p.nd, nd - d0);
        // blocks per value: about 64 for every SM in all
        const int blocks = (int)std::max<long long>(
            1, std::min<long long>((p.units + kDirW - 1) / kDirW, 152 * 64 / ((long long)n * nf)));
        k_rcs_dirs<<<dim3(n, blocks, nf), 32 * kDirW, 0, c->stream>>>(c->nt, geo, c->d_area, work, fk + 2 * f0,
                                                                      dirs + 6 * (size_t)d0, nbc, p.nb, p.units,
                                                                      rcs_m(c), part);
        AIM_CHECK_LAUNCH();
        k_rcs_finish<<<dim3((n + kT / 32 - 1) / (kT / 32), nbc, nf), kT, 0, c->stream>>>(
            n, nd, p.units, nb, b0, p.nb, fk + 2 * f0, part, sig + (size_t)f0 * nb * nd + d0);
        AIM_CHECK_LAUNCH();
      }
    }
}
