// Excitation from envelope samples, far-field envelopes, and their adjoints: the
// pieces that turn the march of Eq. 5 into a differentiable map from incident-envelope
// samples to a far-field objective.  (The paper has no adjoint; these operators are
// the linear maps around its march.)
//
//  * incident envelope e(tau) = sum_i a_i T(tau/dt - i) (the CPPIF of Eq. 3 as the
//    interpolant of the samples a_i), plane wave p e(t - r.k/c) e^{-j k_c r.k}; tested
//    as in Eq. 4:  V_l[k] = sum_i a_i <S_k, p (DT)(l - i - r.k/(c dt)) e^{-j k_c r.k}>,
//    (DT)(u) = T'(u)/dt + j w_c T(u);
//  * far-field envelope in direction r, transverse unit vectors e_1, e_2:
//    F_q(n) = -mu/(4 pi) sum_l sum_k I_l[k] int S_k.e_q (DT)(n - l + r.r'/(c dt))
//             e^{+j k_c r.r'} dS'.
// Every sum runs over the Cowper 7-point cubature of the two triangles of each RWG;
// for each cubature point only the Q+1 time indices inside the support of T
// contribute, so no tap table is stored.
#include <algorithm>
#include <cmath>
#include <vector>

#include "aim_internal.h"
#include "tbasis.cuh"

namespace {

constexpr int kT = 256;

struct WaveArgs {
  double kx, ky, kz, px, py, pz;
};

struct DirArgs {
  int nd;
  const double* r;   // [nd][3]
  const double* e1;  // [nd][3]
  const double* e2;  // [nd][3]
};

struct MeshArgs {
  const int* rtri;
  const int* rfree;
  const double* len;
  const double* area;
  const double* V;
  const double* qp;
  const double* qw;
  int ns;
  double dt, wc, kc, cdt;
  double mu;  // permeability of the background medium
  TBasis tb;
};

__device__ __forceinline__ double2 dt_basis(const MeshArgs& m, double v) {  // (DT)(v)
  double T[4];
  cppif_eval(m.tb, v, T);
  return make_double2(T[1] / m.dt, m.wc * T[0]);
}

__device__ __forceinline__ double2 cm(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmc(double2 a, double2 b) {  // conj(a) b
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// V_l[k], l = l0..l0+n_steps-1 into out[l - l0] (thread per (l, k))
__global__ void __launch_bounds__(kT) k_exc_samples(MeshArgs m, WaveArgs w, int i0, int n_samp,
                                                    const double2* __restrict__ a, int l0, int n_steps,
                                                    double2* __restrict__ out) {
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)n_steps * m.ns) return;
  const int l = (int)(idx / m.ns) + l0, k = (int)(idx % m.ns);
  double2 acc = make_double2(0, 0);
  for (int side = 0; side < 2; ++side) {
    const int t = m.rtri[2 * k + side];
    const double* vf = m.V + 3 * m.rfree[2 * k + side];
    const double cS = (side == 0 ? 1.0 : -1.0) * m.len[k] / (2.0 * m.area[t]);
    for (int q = 0; q < 7; ++q) {
      const double* r = m.qp + 21 * t + 3 * q;
      const double rk = r[0] * w.kx + r[1] * w.ky + r[2] * w.kz;
      const double u = rk / m.cdt;
      double s, c;
      sincos(-m.kc * rk, &s, &c);
      const double sp = cS * ((r[0] - vf[0]) * w.px + (r[1] - vf[1]) * w.py + (r[2] - vf[2]) * w.pz);
      const double wt = m.qw[7 * t + q] * sp;
      const int ilo = max(i0, (int)floor(l - u - m.tb.Q)), ihi = min(i0 + n_samp - 1, (int)ceil(l - u + 1));
      double2 sum = make_double2(0, 0);
      for (int i = ilo; i <= ihi; ++i) {
        const double2 f = dt_basis(m, l - i - u);
        const double2 p = cm(f, a[i - i0]);
        sum.x += p.x;
        sum.y += p.y;
      }
      const double2 e = cm(sum, make_double2(c, s));
      acc.x += wt * e.x;
      acc.y += wt * e.y;
    }
  }
  out[(size_t)(l - l0) * m.ns + k] = acc;
}

template <class T>
__device__ __forceinline__ T wsum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double2 block_sum(double2 v) {
  __shared__ double red[2][kT / 32];
  v.x = wsum(v.x);
  v.y = wsum(v.y);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = v.x;
    red[1][threadIdx.x >> 5] = v.y;
  }
  __syncthreads();
  double2 s = make_double2(0, 0);
  if (threadIdx.x == 0)
    for (int q = 0; q < kT / 32; ++q) {
      s.x += red[0][q];
      s.y += red[1][q];
    }
  __syncthreads();
  return s;
}

// grad_i (+)= sum_l sum_k conj(B_{l-i}[k]) lam_l[k] over l = l0..l0+n_steps-1, lam_l =
// lam[l - l0] (or its conjugate with conj_lam); block per sample i = i0 + blockIdx.x
__global__ void __launch_bounds__(kT) k_exc_samples_adj(MeshArgs m, WaveArgs w, int i0, int l0, int n_steps,
                                                        const double2* __restrict__ lam, int conj_lam, int accumulate,
                                                        double2* __restrict__ grad) {
  const int i = i0 + blockIdx.x;
  double2 acc = make_double2(0, 0);
  for (int k = threadIdx.x; k < m.ns; k += blockDim.x) {
    for (int side = 0; side < 2; ++side) {
      const int t = m.rtri[2 * k + side];
      const double* vf = m.V + 3 * m.rfree[2 * k + side];
      const double cS = (side == 0 ? 1.0 : -1.0) * m.len[k] / (2.0 * m.area[t]);
      for (int q = 0; q < 7; ++q) {
        const double* r = m.qp + 21 * t + 3 * q;
        const double rk = r[0] * w.kx + r[1] * w.ky + r[2] * w.kz;
        const double u = rk / m.cdt;
        double s, c;
        sincos(-m.kc * rk, &s, &c);
        const double sp = cS * ((r[0] - vf[0]) * w.px + (r[1] - vf[1]) * w.py + (r[2] - vf[2]) * w.pz);
        const double wt = m.qw[7 * t + q] * sp;
        const int llo = max(l0, (int)floor(i + u - 1)), lhi = min(l0 + n_steps - 1, (int)ceil(i + u + m.tb.Q));
        for (int l = llo; l <= lhi; ++l) {
          const double2 f = cm(dt_basis(m, l - i - u), make_double2(c, s));
          double2 lv = lam[(size_t)(l - l0) * m.ns + k];
          if (conj_lam) lv.y = -lv.y;
          const double2 p = cmc(f, lv);
          acc.x += wt * p.x;
          acc.y += wt * p.y;
        }
      }
    }
  }
  const double2 sum = block_sum(acc);
  if (threadIdx.x == 0) {
    if (accumulate) {
      grad[blockIdx.x].x += sum.x;
      grad[blockIdx.x].y += sum.y;
    } else {
      grad[blockIdx.x] = sum;
    }
  }
}

// F[n - n0][d][q] (+)= the contribution of I_l, l = l0..l0+n_steps-1 (I_l = I[l - l0]), for
// n = n1..n1+gridDim.x/nd-1 (block per (n, d))
__global__ void __launch_bounds__(kT) k_farfield(MeshArgs m, DirArgs d, int l0, int n_steps,
                                                 const double2* __restrict__ I, int n0, int n1, int accumulate,
                                                 double2* __restrict__ F) {
  const int n = n1 + blockIdx.x / d.nd, di = blockIdx.x % d.nd;
  const double* rh = d.r + 3 * di;
  const double* e1 = d.e1 + 3 * di;
  const double* e2 = d.e2 + 3 * di;
  double2 a1 = make_double2(0, 0), a2 = make_double2(0, 0);
  for (int k = threadIdx.x; k < m.ns; k += blockDim.x) {
    for (int side = 0; side < 2; ++side) {
      const int t = m.rtri[2 * k + side];
      const double* vf = m.V + 3 * m.rfree[2 * k + side];
      const double cS = (side == 0 ? 1.0 : -1.0) * m.len[k] / (2.0 * m.area[t]);
      for (int q = 0; q < 7; ++q) {
        const double* r = m.qp + 21 * t + 3 * q;
        const double rr = r[0] * rh[0] + r[1] * rh[1] + r[2] * rh[2];
        const double wv = rr / m.cdt;
        double s, c;
        sincos(m.kc * rr, &s, &c);
        const double sx = cS * (r[0] - vf[0]), sy = cS * (r[1] - vf[1]), sz = cS * (r[2] - vf[2]);
        const double p1 = m.qw[7 * t + q] * (sx * e1[0] + sy * e1[1] + sz * e1[2]);
        const double p2 = m.qw[7 * t + q] * (sx * e2[0] + sy * e2[1] + sz * e2[2]);
        const int llo = max(l0, (int)floor(n + wv - m.tb.Q)), lhi = min(l0 + n_steps - 1, (int)ceil(n + wv + 1));
        double2 sum = make_double2(0, 0);
        for (int l = llo; l <= lhi; ++l) {
          const double2 p = cm(dt_basis(m, n - l + wv), I[(size_t)(l - l0) * m.ns + k]);
          sum.x += p.x;
          sum.y += p.y;
        }
        const double2 e = cm(sum, make_double2(c, s));
        a1.x += p1 * e.x;
        a1.y += p1 * e.y;
        a2.x += p2 * e.x;
        a2.y += p2 * e.y;
      }
    }
  }
  const double cf = -m.mu / (4.0 * aimc::kPi);
  const double2 s1 = block_sum(a1);
  const double2 s2 = block_sum(a2);
  if (threadIdx.x == 0) {
    double2* f = F + ((size_t)(n - n0) * d.nd + di) * 2;
    if (accumulate) {
      f[0].x += cf * s1.x;
      f[0].y += cf * s1.y;
      f[1].x += cf * s2.x;
      f[1].y += cf * s2.y;
    } else {
      f[0] = make_double2(cf * s1.x, cf * s1.y);
      f[1] = make_double2(cf * s2.x, cf * s2.y);
    }
  }
}

// G_l[k] = conj(-mu/4pi) sum_n sum_{d,q} conj(A_{n-l}[d][q][k]) F[n][d][q] for l = l0..l0+n_steps-1
// into G[l - l0] (conjugated with conj_out); thread per (l, k)
__global__ void __launch_bounds__(kT) k_farfield_adj(MeshArgs m, DirArgs d, int l0, int n_steps, int n0, int n_out,
                                                     const double2* __restrict__ F, int conj_out,
                                                     double2* __restrict__ G) {
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)n_steps * m.ns) return;
  const int l = (int)(idx / m.ns) + l0, k = (int)(idx % m.ns);
  double2 acc = make_double2(0, 0);
  for (int di = 0; di < d.nd; ++di) {
    const double* rh = d.r + 3 * di;
    const double* e1 = d.e1 + 3 * di;
    const double* e2 = d.e2 + 3 * di;
    for (int side = 0; side < 2; ++side) {
      const int t = m.rtri[2 * k + side];
      const double* vf = m.V + 3 * m.rfree[2 * k + side];
      const double cS = (side == 0 ? 1.0 : -1.0) * m.len[k] / (2.0 * m.area[t]);
      for (int q = 0; q < 7; ++q) {
        const double* r = m.qp + 21 * t + 3 * q;
        const double rr = r[0] * rh[0] + r[1] * rh[1] + r[2] * rh[2];
        const double wv = rr / m.cdt;
        double s, c;
        sincos(m.kc * rr, &s, &c);
        const double sx = cS * (r[0] - vf[0]), sy = cS * (r[1] - vf[1]), sz = cS * (r[2] - vf[2]);
        const double p1 = m.qw[7 * t + q] * (sx * e1[0] + sy * e1[1] + sz * e1[2]);
        const double p2 = m.qw[7 * t + q] * (sx * e2[0] + sy * e2[1] + sz * e2[2]);
        const int nlo = max(n0, (int)floor(l - wv - 1)), nhi = min(n0 + n_out - 1, (int)ceil(l - wv + m.tb.Q));
        for (int n = nlo; n <= nhi; ++n) {
          const double2 f = cm(dt_basis(m, n - l + wv), make_double2(c, s));
          const double2* Fn = F + ((size_t)(n - n0) * d.nd + di) * 2;
          const double2 u1 = cmc(f, Fn[0]), u2 = cmc(f, Fn[1]);
          acc.x += p1 * u1.x + p2 * u2.x;
          acc.y += p1 * u1.y + p2 * u2.y;
        }
      }
    }
  }
  const double cf = -m.mu / (4.0 * aimc::kPi);  // real: conj(cf) = cf
  G[(size_t)(l - l0) * m.ns + k] = make_double2(cf * acc.x, conj_out ? -cf * acc.y : cf * acc.y);
}

// ---------------------------------------------------------------- far field through taps
// The coefficient of I_l[k] in F[n][d][q] depends on n - l only, and is non-zero for the few
// shifts s = n - l with s + r.r'/(c dt) in (-1, Q] for some cubature point of the RWG:
//   A_s[q] = sum_points p_q (DT)(s + w) e^{j k_c r.r'},  F[n] = sum_{k,s} A_s[k] I_{n-s}[k].
// Both directions therefore form the taps of a tile of (RWG, direction) pairs once, in
// shared memory, and run the time sums from them, instead of evaluating the basis and the
// phase at every point for every n (or l).  Bound by FP64 arithmetic: per (RWG, direction)
// about 14 x 110 operations for the taps and 8 per shift and step of the time sum.  (60
// steps, 16 directions, 1920 RWGs, far field and adjoint: 24.5 ms before, 0.95 ms now.)
constexpr int kMaxTaps = 8;      // shifts held per pair
constexpr int kFarK = 32, kFarD = 4, kFarN = 64;    // far field: RWGs, directions, times per block
constexpr int kAdjK = 8, kAdjD = 16, kAdjL = 64;    // adjoint: RWGs, directions per tile, steps per block
constexpr int kPairs = kT / 2;   // pairs of a tile: two lanes (the two faces) each
static_assert(kFarK * kFarD == kPairs && kAdjK * kAdjD == kPairs && kFarN * kFarD == kT, "tile shapes");

struct TapCoef {  // T and T' of the pieces: T = sum coef[p] u^p, T' = sum dcoef[p] u^(p-1)
  double c[aimc::kMaxOrder + 1][aimc::kMaxOrder + 1], d[aimc::kMaxOrder + 1][aimc::kMaxOrder + 1];
};
__device__ __forceinline__ void load_coef(const MeshArgs& m, TapCoef& tc) {
  for (int i = threadIdx.x; i < (aimc::kMaxOrder + 1) * (aimc::kMaxOrder + 1); i += kT) {
    const int j = i / (aimc::kMaxOrder + 1), p = i % (aimc::kMaxOrder + 1);
    tc.c[j][p] = m.tb.coef[j][p];
    tc.d[j][p] = p * m.tb.coef[j][p];
  }
}

// the taps of the pair (k, direction d); lanes 2i and 2i + 1 take its two faces.  The first
// shift goes to first->s, taps first .. first + nt - 1 to A[i][q] (zeros for an invalid pair),
// and bit i of first->hit says whether a point lies in the support of tap i: the others are
// left out of the time sums, where a zero times an infinity would spoil times that the pair
// does not reach.
struct FirstTap {
  int s;
  unsigned hit;
};
__device__ __forceinline__ void far_taps(const MeshArgs& m, const TapCoef& tc, const DirArgs& d, int k, int di,
                                         bool valid, int nt, double2* A, FirstTap* first) {
  const int side = threadIdx.x & 1, Q = m.tb.Q;
  double2 a1[kMaxTaps] = {}, a2[kMaxTaps] = {};
  double w[7], p1[7], p2[7];
  double wmax = -1e300;
  if (valid) {
    const double *rh = d.r + 3 * di, *e1 = d.e1 + 3 * di, *e2 = d.e2 + 3 * di;
    const int t = m.rtri[2 * k + side];
    const double* vf = m.V + 3 * m.rfree[2 * k + side];
    const double cS = (side == 0 ? 1.0 : -1.0) * m.len[k] / (2.0 * m.area[t]);
    for (int q = 0; q < 7; ++q) {
      const double* r = m.qp + 21 * t + 3 * q;
      const double sx = r[0] - vf[0], sy = r[1] - vf[1], sz = r[2] - vf[2], wq = cS * m.qw[7 * t + q];
      w[q] = r[0] * rh[0] + r[1] * rh[1] + r[2] * rh[2];
      p1[q] = wq * (sx * e1[0] + sy * e1[1] + sz * e1[2]);
      p2[q] = wq * (sx * e2[0] + sy * e2[1] + sz * e2[2]);
    }
    for (int q = 0; q < 7; ++q) wmax = fmax(wmax, w[q]);
  }
  wmax = fmax(wmax, __shfl_xor_sync(0xffffffffu, wmax, 1)) / m.cdt;
  const int s0 = valid ? (int)floor(-1.0 - wmax) + 1 : 0;
  unsigned hit = 0;
  if (valid) {
    const double idt = 1.0 / m.dt;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      double sn, cs;
      sincos(m.kc * w[q], &sn, &cs);
      const double wv = w[q] / m.cdt;
      const double2 g1 = make_double2(p1[q] * cs, p1[q] * sn), g2 = make_double2(p2[q] * cs, p2[q] * sn);
#pragma unroll
      for (int i = 0; i < kMaxTaps; ++i) {
        const double v = (s0 + i) + wv, jr = ceil(v);
        if (i < nt && jr >= 0.0 && jr <= (double)Q) {
          const int j = (int)jr;
          hit |= 1u << i;
          double T = 0, D = 0;
          for (int p = Q; p >= 0; --p) T = T * v + tc.c[j][p];
          for (int p = Q; p >= 1; --p) D = D * v + tc.d[j][p];
          const double2 f = make_double2(D * idt, m.wc * T), x = cm(f, g1), y = cm(f, g2);
          a1[i].x += x.x;
          a1[i].y += x.y;
          a2[i].x += y.x;
          a2[i].y += y.y;
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kMaxTaps; ++i)
    if (i < nt) {  // the two faces: lane 0 stores the first polarisation, lane 1 the second
      const double2 mine = side ? a2[i] : a1[i], other = side ? a1[i] : a2[i];
      A[2 * i + side] = make_double2(mine.x + __shfl_xor_sync(0xffffffffu, other.x, 1),
                                     mine.y + __shfl_xor_sync(0xffffffffu, other.y, 1));
    }
  hit |= __shfl_xor_sync(0xffffffffu, hit, 1);
  if (side == 0) *first = FirstTap{s0, hit};
}

// part[split][n - na][d][q] over the RWG tiles of a split (every gridDim.y-th tile: the splits
// depend on the mesh alone, so that a value rounds the same whatever else is in the call);
// grid (direction tiles, splits, time tiles).  I_l = I[l - l0], l = l0 .. l0 + n_steps - 1.
__global__ void __launch_bounds__(kT) k_far_sum(MeshArgs m, DirArgs d, int l0, int n_steps, int taps,
                                                const double2* __restrict__ I, int na, int n_cnt,
                                                double2* __restrict__ part) {
  extern __shared__ double2 tap_smem[];  // [pair][taps][2]
  __shared__ TapCoef tc;
  __shared__ FirstTap first[kPairs];
  load_coef(m, tc);
  __syncthreads();
  const int pair = threadIdx.x >> 1, d0 = blockIdx.x * kFarD;
  const int nn = blockIdx.z * kFarN + threadIdx.x % kFarN, dd = threadIdx.x / kFarN, n = na + nn;
  double2 f1 = make_double2(0, 0), f2 = make_double2(0, 0);
  for (int k0 = blockIdx.y * kFarK; k0 < m.ns; k0 += gridDim.y * kFarK) {
    {
      const int k = k0 + pair % kFarK, di = d0 + pair / kFarK;
      far_taps(m, tc, d, k, di, k < m.ns && di < d.nd, taps, tap_smem + (size_t)pair * taps * 2, first + pair);
    }
    __syncthreads();
    for (int kk = 0; kk < kFarK && k0 + kk < m.ns; ++kk) {
      const double2* A = tap_smem + (size_t)(dd * kFarK + kk) * taps * 2;
      const FirstTap ft = first[dd * kFarK + kk];
      const int l = n - ft.s - l0;  // of the first shift
      for (int i = 0; i < taps; ++i)
        if ((ft.hit >> i & 1) && l - i >= 0 && l - i < n_steps) {
          const double2 x = I[(size_t)(l - i) * m.ns + k0 + kk], u = cm(A[2 * i], x), v = cm(A[2 * i + 1], x);
          f1.x += u.x;
          f1.y += u.y;
          f2.x += v.x;
          f2.y += v.y;
        }
    }
    __syncthreads();
  }
  if (nn < n_cnt && d0 + dd < d.nd) {
    double2* o = part + (((size_t)blockIdx.y * n_cnt + nn) * d.nd + d0 + dd) * 2;
    o[0] = f1;
    o[1] = f2;
  }
}

// F (+)= cf * the sum of the splits, n values of rows of `row`, rows of F `ldf` apart
__global__ void __launch_bounds__(kT) k_far_finish(long long n, int splits, double cf, int accumulate, int row, int ldf,
                                                   const double2* __restrict__ part, double2* __restrict__ F) {
  const long long i = blockIdx.x * (long long)kT + threadIdx.x;
  if (i >= n) return;
  double2 s = make_double2(0, 0);
#pragma unroll 8
  for (int q = 0; q < splits; ++q) {
    s.x += part[q * n + i].x;
    s.y += part[q * n + i].y;
  }
  double2* f = F + (i / row) * ldf + i % row;
  const double2 o = accumulate ? *f : make_double2(0, 0);
  *f = make_double2(o.x + cf * s.x, o.y + cf * s.y);
}

// the adjoint: G_l[k] = cf sum_{n,d,q} conj(A_{n-l}) F[n][d][q]; grid step tiles x RWG tiles,
// the k_tiles RWG tiles fastest (in one dimension: there may be more step tiles than the others hold)
__global__ void __launch_bounds__(kT) k_far_adj(MeshArgs m, DirArgs d, int l0, int n_steps, int taps, int n0, int n_out,
                                                int k_tiles, const double2* __restrict__ F, int conj_out,
                                                double2* __restrict__ G) {
  extern __shared__ double2 tap_smem[];
  __shared__ TapCoef tc;
  __shared__ FirstTap first[kPairs];
  load_coef(m, tc);
  __syncthreads();
  const int pair = threadIdx.x >> 1, k0 = blockIdx.x % k_tiles * kAdjK, lb = blockIdx.x / k_tiles * kAdjL;
  const int kk = threadIdx.x >> 5, ll = threadIdx.x & 31;
  double2 acc[kAdjL / 32] = {};
  for (int d0 = 0; d0 < d.nd; d0 += kAdjD) {
    {
      const int k = k0 + pair % kAdjK, di = d0 + pair / kAdjK;
      far_taps(m, tc, d, k, di, k < m.ns && di < d.nd, taps, tap_smem + (size_t)pair * taps * 2, first + pair);
    }
    __syncthreads();
    for (int dd = 0; dd < kAdjD && d0 + dd < d.nd; ++dd) {
      const double2* A = tap_smem + (size_t)(dd * kAdjK + kk) * taps * 2;
      const FirstTap ft = first[dd * kAdjK + kk];
#pragma unroll
      for (int h = 0; h < kAdjL / 32; ++h) {
        const int n = l0 + lb + ll + 32 * h + ft.s - n0;  // of the first shift
        for (int i = 0; i < taps; ++i)
          if ((ft.hit >> i & 1) && n + i >= 0 && n + i < n_out) {
            const double2* f = F + ((size_t)(n + i) * d.nd + d0 + dd) * 2;
            const double2 u = cmc(A[2 * i], f[0]), v = cmc(A[2 * i + 1], f[1]);
            acc[h].x += u.x + v.x;
            acc[h].y += u.y + v.y;
          }
      }
    }
    __syncthreads();
  }
  const double cf = -m.mu / (4.0 * aimc::kPi);  // real: conj(cf) = cf
#pragma unroll
  for (int h = 0; h < kAdjL / 32; ++h) {
    const int l = lb + ll + 32 * h;
    if (l < n_steps && k0 + kk < m.ns)
      G[(size_t)l * m.ns + k0 + kk] = make_double2(cf * acc[h].x, conj_out ? -cf * acc[h].y : cf * acc[h].y);
  }
}

// valT[m][e] = val[m][perm[e]]: the near-zone values of the transposed matrices
__global__ void k_gather_transpose(int nnz, int nm, const int* __restrict__ perm, const double2* __restrict__ val,
                                   double2* __restrict__ valT) {
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)nnz * nm) return;
  const int e = (int)(idx % nnz), mm = (int)(idx / nnz);
  valT[idx] = val[(size_t)mm * nnz + perm[e]];
}

MeshArgs mesh_args(aim_ctx* c) {
  MeshArgs m;
  m.rtri = c->d_rtri;
  m.rfree = c->d_rfree;
  m.len = c->d_len;
  m.area = c->d_area;
  m.V = c->d_v;
  m.qp = c->d_qp;
  m.qw = c->d_qw;
  m.ns = c->ns;
  m.dt = c->dt;
  m.wc = c->wc;
  m.kc = c->kc;
  m.cdt = c->c_med * c->dt;
  m.mu = c->mu_med;
  if (c->tb.kind != AIM_CPPIF)
    throw AimError{AIM_ERR_ARG, "the sampled-envelope excitation and far field interpolate with the CPPIF only"};
  m.tb = c->tb;
  return m;
}

}  // namespace

// time reach of the cubature points in units of dt: every point r has |r.u| / (c dt) <= this
// for any u no longer than len (the largest vertex distance from the origin bounds the points)
static double reach(aim_ctx* c, double len = 1.0) { return c->rmax * len / (c->c_med * c->dt); }

// shifts an RWG's taps can span: s + w in (-1, Q] with w varying by at most the largest
// distance between two points of an RWG times the direction's length; 0 where that exceeds
// kMaxTaps (RWGs of several c dt: the sums go point by point, k_farfield and k_farfield_adj)
static int tap_count(const aim_ctx* c, double len) {
  const double n = std::floor(c->tb.Q + 2.0 + c->rwg_span * len / (c->c_med * c->dt));
  return n <= kMaxTaps ? (int)n : 0;
}

void adj_excitation_samples(aim_ctx* c, const double* khat, const double* phat, int i0, int n_samp,
                            const double2* a, int l0, int n_steps, double2* V) {
  WaveArgs w{khat[0], khat[1], khat[2], phat[0], phat[1], phat[2]};
  const long long n = (long long)n_steps * c->ns;
  k_exc_samples<<<(int)((n + kT - 1) / kT), kT, 0, c->stream>>>(mesh_args(c), w, i0, n_samp, a, l0, n_steps, V);
  AIM_CHECK_LAUNCH();
}

// grad over the samples i0..i0+n_samp-1; with accumulate only the samples whose taps reach
// steps l0..l0+n_steps-1 are visited (the others receive nothing)
void adj_excitation_samples_adjoint(aim_ctx* c, const double* khat, const double* phat, int i0, int n_samp,
                                    int l0, int n_steps, const double2* lam, bool conj_lam, bool accumulate,
                                    double2* grad) {
  WaveArgs w{khat[0], khat[1], khat[2], phat[0], phat[1], phat[2]};
  int ia = i0, ib = i0 + n_samp - 1;
  if (accumulate) {  // B_{l-i} is non-zero only for l - i - u in (-1, Q], |u| <= reach
    const double u = reach(c);
    ia = std::max(ia, (int)std::floor(l0 - u - c->tb.Q) - 1);
    ib = std::min(ib, (int)std::ceil(l0 + n_steps - 1 + u + 1) + 1);
    if (ib < ia) return;
  }
  k_exc_samples_adj<<<ib - ia + 1, kT, 0, c->stream>>>(mesh_args(c), w, ia, l0, n_steps, lam, conj_lam ? 1 : 0,
                                                     accumulate ? 1 : 0, grad + (ia - i0));
  AIM_CHECK_LAUNCH();
}

// Passes of the far field over nd directions and n_cnt times: the splits of the RWG tiles, of
// the mesh alone (two for every SM where there are as many tiles), and the directions and times
// of a pass, whose partial sums stay within 64 MB.
struct FarPass {
  int splits, nd, n;
  size_t elems;
};
static FarPass far_pass(const aim_ctx* c, int nd, int n_cnt) {
  constexpr long long kCap = (64LL << 20) / sizeof(double2);
  FarPass p;
  p.splits = std::min(304, (c->ns + kFarK - 1) / kFarK);
  const long long per_d = (long long)p.splits * kFarN * 2;  // one direction, one tile of times
  p.nd = per_d * nd <= kCap ? nd : (int)(kCap / per_d / kFarD) * kFarD;
  p.n = (int)std::min<long long>(n_cnt, kCap / (per_d * p.nd) * kFarN);
  p.elems = (size_t)p.splits * p.nd * 2 * p.n;
  return p;
}

// the partial sums that single steps of a march need, at their widest window
void adj_farfield_reserve(aim_ctx* c, const FarDirs& dirs, int n_out) {
  if (tap_count(c, dirs.len) == 0) return;
  const double window = 2.0 * reach(c, dirs.len) + c->tb.Q + 6.0;  // of adj_farfield, one step
  const FarPass p = far_pass(c, dirs.nd, (int)std::min<double>(n_out, window));
  aim_grow(c, c->far_part, c->far_cap, p.elems);
}

// F over n = n0..n0+n_out-1; with accumulate only the n the steps l0..l0+n_steps-1 reach
void adj_farfield(aim_ctx* c, const FarDirs& dirs, int l0, int n_steps, const double2* I, int n0, int n_out,
                  bool accumulate, double2* F) {
  const int nd = dirs.nd;
  DirArgs d{nd, dirs.d, dirs.d + 3 * nd, dirs.d + 6 * nd};
  int na = n0, nb_ = n0 + n_out - 1;
  if (accumulate) {  // A_{n-l} is non-zero only for n - l + w in (-1, Q], |w| <= reach
    const double u = reach(c, dirs.len);
    na = (int)std::max<double>(na, std::floor(l0 - u - 1) - 1);
    nb_ = (int)std::min<double>(nb_, std::ceil(l0 + n_steps - 1 + u + c->tb.Q) + 1);
    if (nb_ < na) return;
  }
  const MeshArgs m = mesh_args(c);
  const int taps = tap_count(c, dirs.len), n_cnt = nb_ - na + 1;
  if (taps == 0) {
    k_farfield<<<n_cnt * nd, kT, 0, c->stream>>>(m, d, l0, n_steps, I, n0, na, accumulate ? 1 : 0, F);
    AIM_CHECK_LAUNCH();
    return;
  }
  const FarPass p = far_pass(c, nd, n_cnt);
  aim_grow(c, c->far_part, c->far_cap, p.elems);
  for (int d0 = 0; d0 < nd; d0 += p.nd)
    for (int i0 = 0; i0 < n_cnt; i0 += p.n) {
      const int pd = std::min(p.nd, nd - d0), pn = std::min(p.n, n_cnt - i0);
      const DirArgs dp{pd, d.r + 3 * (size_t)d0, d.e1 + 3 * (size_t)d0, d.e2 + 3 * (size_t)d0};
      k_far_sum<<<dim3((pd + kFarD - 1) / kFarD, p.splits, (pn + kFarN - 1) / kFarN), kT,
                  kPairs * taps * 2 * sizeof(double2), c->stream>>>(m, dp, l0, n_steps, taps, I, na + i0, pn,
                                                                    c->far_part);
      AIM_CHECK_LAUNCH();
      const long long n = (long long)pn * pd * 2;
      k_far_finish<<<(int)((n + kT - 1) / kT), kT, 0, c->stream>>>(
          n, p.splits, -m.mu / (4.0 * aimc::kPi), accumulate ? 1 : 0, 2 * pd, 2 * nd, c->far_part,
          F + ((size_t)(na + i0 - n0) * nd + d0) * 2);
      AIM_CHECK_LAUNCH();
    }
}

void adj_farfield_adjoint(aim_ctx* c, const FarDirs& dirs, int l0, int n_steps, int n0, int n_out,
                          const double2* F, bool conj_out, double2* G) {
  const int nd = dirs.nd;
  DirArgs d{nd, dirs.d, dirs.d + 3 * nd, dirs.d + 6 * nd};
  if (const int taps = tap_count(c, dirs.len)) {
    const int k_tiles = (c->ns + kAdjK - 1) / kAdjK;
    const long long blocks = (long long)k_tiles * ((n_steps + (long long)kAdjL - 1) / kAdjL);
    k_far_adj<<<(unsigned)blocks, kT, kPairs * taps * 2 * sizeof(double2), c->stream>>>(
        mesh_args(c), d, l0, n_steps, taps, n0, n_out, k_tiles, F, conj_out ? 1 : 0, G);
    AIM_CHECK_LAUNCH();
    return;
  }
  const long long n = (long long)n_steps * c->ns;
  k_farfield_adj<<<(int)((n + kT - 1) / kT), kT, 0, c->stream>>>(mesh_args(c), d, l0, n_steps, n0, n_out, F,
                                                                conj_out ? 1 : 0, G);
  AIM_CHECK_LAUNCH();
}

// transposed near-zone values (same pattern: the near relation is symmetric)
void adj_ensure_near_transpose(aim_ctx* c) {
  if (c->d_nearT || c->nnz == 0) return;
  const int ns = c->ns;
  const long long nnz = c->nnz;
  std::vector<int> perm(nnz);
  for (int k = 0; k < ns; ++k)
    for (int e = c->h_rowptr[k]; e < c->h_rowptr[k + 1]; ++e) {
      const int j = c->h_col[e];
      const int* b = c->h_col.data() + c->h_rowptr[j];
      const int* en = c->h_col.data() + c->h_rowptr[j + 1];
      const int* f = std::lower_bound(b, en, k);
      if (f == en || *f != k) throw AimError{AIM_ERR_ARG, "near-zone pattern is not symmetric"};
      perm[e] = (int)(f - c->h_col.data());
    }
  const int nm = c->n_delays + 1;
  int* d_perm = (int*)aim_alloc(c, nnz * sizeof(int));
  c->d_nearT = (double2*)aim_alloc(c, (size_t)nm * nnz * sizeof(double2));
  AIM_CUDA(cudaMemcpyAsync(d_perm, perm.data(), nnz * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  const long long n = nnz * nm;
  k_gather_transpose<<<(int)((n + kT - 1) / kT), kT, 0, c->stream>>>((int)nnz, nm, d_perm, c->d_near, c->d_nearT);
  AIM_CHECK_LAUNCH();
  AIM_CUDA(cudaStreamSynchronize(c->stream));
}
