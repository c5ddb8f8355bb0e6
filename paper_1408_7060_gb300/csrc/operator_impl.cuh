// The ET-AIM operator on the device (Eq. 5, Sec. 4 stages i-iv), templated on the
// complex type of the grid stages (float2: complex64 path, double2: plain path).
//
// Data layout per right-hand side b and component c (x, y, z, div), with L = 2N and the
// nz z-planes z0 .. z0 + nz - 1 of the active box (the nodes some stencil touches):
//   A  [b][c][nz][y<N][x<L]   after anterpolation + forward x-FFT
//   Bf [b][c][nz][y<L][x<L]   after the forward y-FFT (the slab)
//   P  [b][c][nz][y<N][x<N]   potentials after the inverse passes
// The forward z-FFT (length LZ >= 2 nz), the pointwise kernel product and the inverse
// z-FFT are one kernel per column (k_zconv_p2, k_zwarp), so no 3-D spectrum reaches
// memory.  Where a kx plane fits shared memory (plane.cuh) A is kx-major, [b][c][x<L][nz][y<N],
// and the y passes join that kernel: Bf is not used.  Zero padding is pruned in every pass: forward passes read only the non-zero
// inputs, inverse passes write only the needed outputs.
#pragma once
#include <algorithm>
#include <functional>
#include <type_traits>
#include <vector>

#include "aim_internal.h"
#include "fft_kernels.cuh"
#include "operator.h"
#include "plane.cuh"
#include "tma.cuh"

template <class C> struct Real;
template <> struct Real<float2> { using T = float; using F4 = float4; };
template <> struct Real<double2> { using T = double; using F4 = double4_32a; };

template <class C> __device__ __forceinline__ C cvt(double2 a);
template <> __device__ __forceinline__ float2 cvt<float2>(double2 a) { return make_float2((float)a.x, (float)a.y); }
template <> __device__ __forceinline__ double2 cvt<double2>(double2 a) { return a; }

// ---------------------------------------------------------------- stage i + x pass
// radix split of the x passes
__host__ __device__ constexpr int x_r1(int L) { return L == 768 ? 32 : pl_r1(L); }
__host__ __device__ constexpr int x_r2(int L) { return L / x_r1(L); }
// elements between the rows of an x tile: R1 blocks of R2 + 1; kx-major stores take YB rows
// in consecutive lanes, so the pitch is 16 / YB mod 16 (no bank conflict between them)
__host__ __device__ constexpr int x_pitch(int L, int yb) {
  int p = x_r1(L) * (x_r2(L) + 1);
  while (p % 16 != (yb >= 16 ? 1 : yb == 1 ? 0 : 16 / yb)) ++p;
  return p;
}
// S_c[n] = sum_k L_c[n,k] x_k gathered node by node (the transpose of the interpolation
// rows), then the forward x-FFT of each grid row.  One block holds the 4 components of YB
// consecutive rows y of one plane z for BB right-hand sides.  Only the nodes some stencil
// touches are visited (arow: their range per box row, anode: y N + x, aptr: their CSR
// entries); the operator input is interleaved, xs[k][b], so the BB lanes of a node share
// its coefficients and gather adjacent values.  With one right-hand side 4 lanes share a
// node's entries instead (each is an index, coefficient, gather chain).  Both sum a node's
// entries in the same order (entry e into partial sum e mod 4, then (0 + 2) + (1 + 3)), so a
// right-hand side's result does not depend on the batch it is in.  KXM stores the kx-major grid of the plane
// kernel, A[b][c][kx][z][y - ylo] (rows beyond the box written as zeros up to N), runs of
// YB values; otherwise A[b][c][z][y][kx].
template <int L, int YB, int BB, bool KXM, class C>
__global__ void __launch_bounds__(256) k_anterp(const int* __restrict__ arow, const int* __restrict__ anode,
                                                const int* __restrict__ aptr, const int* __restrict__ nidx,
                                                const typename Real<C>::F4* __restrict__ ncoef,
                                                const C* __restrict__ xs, const int* __restrict__ active, int nb,
                                                C* __restrict__ A, const C* __restrict__ twg, int ylo, int nyb, int nz) {
  using R = typename Real<C>::T;
  constexpr int N = L / 2, R1 = x_r1(L), R2 = x_r2(L), PX = x_pitch(L, KXM ? YB : 1), ROWS = 4 * YB * BB;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* in = tw + kTw2<R1, R2>;  // [bs][c][yy][N]
  C* tmp = in + ROWS * N;     // [bs][c][yy][PX]
  load_twiddles2<R1, R2>(tw, twg);
  for (int i = threadIdx.x; i < ROWS * N; i += 256) in[i] = C{};
  pdl_wait();
  const int b0 = blockIdx.x * BB, y0 = blockIdx.y * YB, z = blockIdx.z;  // y relative to the box
  if (BB == 1 && active && !active[b0]) return;
  __syncthreads();
  const int ye = min(y0 + YB, nyb);
  if (y0 < nyb) {
    constexpr int EL = BB == 1 ? 4 : 1;  // lanes per node
    const int k0 = arow[z * nyb + y0], items = (arow[z * nyb + ye] - k0) * (BB * EL);
    // (whole warps run every round, for the sums over the lanes of a node)
    for (int i = threadIdx.x; i - (int)(threadIdx.x & 31) < items; i += 256) {
      const int bs = i % BB, k = min(k0 + i / (BB * EL), k0 + items / (BB * EL) - 1), b = b0 + bs;
      const bool on = i < items && (BB == 1 || (b < nb && !(active && !active[b])));
      const int nd = anode[k], yy = nd / N - ylo - y0, x = nd % N;
      const C* vb = xs + b;
      constexpr int NA = 4 / EL;  // partial sums of a lane
      C a[NA][4] = {};
      auto add = [&](C* t, const typename Real<C>::F4& w, const C& xv) {
        t[0] += (R)w.x * xv;
        t[1] += (R)w.y * xv;
        t[2] += (R)w.z * xv;
        t[3] += (R)w.w * xv;
      };
      int e = on ? aptr[k] + (EL > 1 ? i % EL : 0) : 0;
      const int e1 = on ? aptr[k + 1] : 0;
      // four entries at a time: their index and coefficient loads, then their gathers of
      // x, are independent and in flight together
      for (; e + 3 * EL < e1; e += 4 * EL) {
        int j[4];
        typename Real<C>::F4 w[4];
        C xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          j[u] = nidx[e + u * EL];
          w[u] = ncoef[e + u * EL];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) xv[u] = vb[(size_t)j[u] * nb];
#pragma unroll
        for (int u = 0; u < 4; ++u) add(a[u % NA], w[u], xv[u]);
      }
      if constexpr (EL == 4) {
        for (; e < e1; e += EL) add(a[0], ncoef[e], vb[(size_t)nidx[e] * nb]);
      } else {  // at most 3 are left
#pragma unroll
        for (int u = 0; u < 3; ++u)
          if (e + u < e1) add(a[u], ncoef[e + u], vb[(size_t)nidx[e + u] * nb]);
      }
      if constexpr (EL == 4) {  // lane q of the four keeps component q
        const bool hi = i & 2, od = i & 1;
        C u0 = hi ? a[0][2] : a[0][0], u1 = hi ? a[0][3] : a[0][1];
        const C s0 = hi ? a[0][0] : a[0][2], s1 = hi ? a[0][1] : a[0][3];
        u0.x += __shfl_xor_sync(0xffffffffu, s0.x, 2);
        u0.y += __shfl_xor_sync(0xffffffffu, s0.y, 2);
        u1.x += __shfl_xor_sync(0xffffffffu, s1.x, 2);
        u1.y += __shfl_xor_sync(0xffffffffu, s1.y, 2);
        C t = od ? u1 : u0;
        const C s = od ? u0 : u1;
        t.x += __shfl_xor_sync(0xffffffffu, s.x, 1);
        t.y += __shfl_xor_sync(0xffffffffu, s.y, 1);
        if (on) in[((i & 3) * YB + yy) * N + x] = t;
      } else if (on) {
        C* t = in + (bs * 4 * YB + yy) * N + x;
#pragma unroll
        for (int c = 0; c < 4; ++c) t[c * YB * N] = (a[0][c] + a[2][c]) + (a[1][c] + a[3][c]);
      }
    }
  }
  __syncthreads();
  for (int u = threadIdx.x; u < ROWS * R2; u += 256) {
    const int n2 = u % R2, row = u / R2;
    C v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1 / 2; ++n1) v[n1] = in[row * N + R2 * n1 + n2];
    dft_half_in<R1, L, false, C>(v, tw);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) tmp[row * PX + k1 * (R2 + 1) + n2] = k1 ? v[k1] * tw[k1 * (R2 + 1) + n2] : v[k1];
  }
  __syncthreads();
  for (int u = threadIdx.x; u < ROWS * R1; u += 256) {
    int k1, row;
    if (KXM) {
      const int yy = u % YB, r = u / YB;
      k1 = r % R1;
      row = (r / R1) * YB + yy;
    } else {
      k1 = u % R1;
      row = u / R1;
    }
    const int yy = row % YB, c = (row / YB) & 3, b = b0 + row / (4 * YB);
    if (BB > 1 && (b >= nb || (active && !active[b]))) continue;
    C v[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = tmp[row * PX + k1 * (R2 + 1) + n2];
    DFTL<R2, L, false, C>::run(v, tw);
    if (KXM) {
      C* dst = A + ((size_t)(b * 4 + c) * L * nz + z) * N + y0 + yy;
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) dst[(size_t)(k1 + R1 * k2) * nz * N] = v[k2];
    } else if (y0 + yy < nyb) {
      C* dst = A + (((size_t)(b * 4 + c) * nz + z) * N + ylo + y0 + yy) * L + k1;
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) dst[R1 * k2] = v[k2];
    }
  }
}

// Inverse x-FFT of the kx-major grid: A[bc][kx][z][y] -> P[bc][z][ylo + y][x < N].  One
// block takes YB rows y of one plane z; lanes walk the rows first, so every load is a run
// of YB values, and only the outputs x < N are formed.
template <int L, int YB, class C>
__global__ void __launch_bounds__(256) k_xinv(const C* __restrict__ A, C* __restrict__ P,
                                              const C* __restrict__ twg, int ylo, int nyb, int nz) {
  constexpr int N = L / 2, R1 = x_r1(L), R2 = x_r2(L), PX = x_pitch(L, YB);
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* tmp = tw + kTw2<R1, R2>;
  load_twiddles2<R1, R2>(tw, twg);
  pdl_wait();
  __syncthreads();
  const int y0 = blockIdx.x * YB, z = blockIdx.y, bc = blockIdx.z;
  const C* src = A + ((size_t)bc * L * nz + z) * N + y0;
  for (int u = threadIdx.x; u < YB * R2; u += 256) {
    const int yy = u % YB, n2 = u / YB;
    C v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) v[n1] = src[(size_t)(R2 * n1 + n2) * nz * N + yy];
    DFTL<R1, L, true, C>::run(v, tw);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1)
      tmp[yy * PX + k1 * (R2 + 1) + n2] = k1 ? v[k1] * conjc(tw[k1 * (R2 + 1) + n2]) : v[k1];
  }
  __syncthreads();
  C* dst = P + ((size_t)bc * nz + z) * N * N + (size_t)(ylo + y0) * N;
  for (int u = threadIdx.x; u < YB * R1; u += 256) {
    const int k1 = u % R1, yy = u / R1;
    C v[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = tmp[yy * PX + k1 * (R2 + 1) + n2];
    dft_half_out<R2, L, true, C>(v, tw);
    if (y0 + yy < nyb)
#pragma unroll
      for (int k2 = 0; k2 < R2 / 2; ++k2) dst[(size_t)yy * N + k1 + R1 * k2] = v[k2];
  }
}

// Operator input: x_b = scale_b(j) * dinv .* v_b (selection, Krylov scale and
// preconditioner applied once), in the grid precision for the anterpolation gather
// (interleaved, xs[k][b]) and in FP64 for the near-zone product (xd[b][k]).
template <class C>
__global__ void __launch_bounds__(256) k_prep(const double2* __restrict__ v, const double2* __restrict__ dinv,
                                              VecSel vs, const int* __restrict__ active, int ns, int nb,
                                              C* __restrict__ xs, double2* __restrict__ xd) {
  pdl_wait();
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)nb * ns) return;
  const int b = (int)(idx / ns), k = (int)(idx % ns);
  if (active && !active[b]) return;
  double sc = 1.0;
  if (vs.sel) {
    const int j = *vs.sel + vs.off;
    v += j * vs.stride;
    if (vs.scale) sc = vs.scale[b * 64 + j];
  }
  double2 x = v[idx];
  x = make_double2(sc * x.x, sc * x.y);
  if (dinv) {
    const double2 d = dinv[k];
    x = make_double2(x.x * d.x - x.y * d.y, x.x * d.y + x.y * d.x);
  }
  xs[(size_t)k * nb + b] = cvt<C>(x);
  if (xd) xd[idx] = x;
}

// The same with the SAI as the preconditioner: x_b[k] = scale_b(j) *
// sum_e M[k, col_e] v_b[col_e] over row k of its CSR pattern (at most 144 entries).  16
// lanes per row (two rows per warp), fixed-order butterfly sum over the 16 lanes.  M is
// applied in the grid precision: complex64 (M rounded to FP32, products and sums in FP32,
// like the grid stages it feeds) or complex128 (FP64).
template <class C>
__global__ void __launch_bounds__(256) k_prep_sai(const double2* __restrict__ v, const float2* __restrict__ vf,
                                                  const C* __restrict__ sai, const int* __restrict__ rowptr,
                                                  const int* __restrict__ col, VecSel vs,
                                                  const int* __restrict__ active, int ns, int nb,
                                                  C* __restrict__ xs, double2* __restrict__ xd) {
  pdl_wait();
  using R = typename Real<C>::T;
  const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 4;
  const int lane = threadIdx.x & 15;
  const bool valid = w < (long long)nb * ns;  // both rows of a warp join the shuffles
  const int b = valid ? (int)(w / ns) : 0, k = valid ? (int)(w % ns) : 0;
  const bool on = valid && !(active && !active[b]);
  double sc = 1.0;
  if (vs.sel) {
    const int j = *vs.sel + vs.off;
    v += j * vs.stride;
    if (vs.scale) sc = vs.scale[b * 64 + j];
  }
  const double2* vb = v + (size_t)b * ns;
  R xr = 0, xi = 0;
  if (on) {
    // up to 9 entries per lane: indices and values first, then the gathered vector
    // entries, then the products in entry order
    const int e0 = rowptr[k] + lane, e1 = rowptr[k + 1];
    int j[9];
    C m[9];
    double2 u[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const int e = e0 + 16 * q;
      j[q] = e < e1 ? col[e] : -1;
      m[q] = e < e1 ? sai[e] : C{};
    }
    if (vf) {  // complex64 copy of v_j: no FP64 -> FP32 conversion per gathered entry
      const float2* vfb = vf + (size_t)b * ns;
      float2 uf[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) uf[q] = j[q] >= 0 ? vfb[j[q]] : make_float2(0, 0);
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (j[q] >= 0) {
          const R ur = (R)uf[q].x, ui = (R)uf[q].y;
          xr += m[q].x * ur - m[q].y * ui;
          xi += m[q].x * ui + m[q].y * ur;
        }
    } else {
#pragma unroll
      for (int q = 0; q < 9; ++q) u[q] = j[q] >= 0 ? vb[j[q]] : make_double2(0, 0);
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (j[q] >= 0) {
          const R ur = (R)u[q].x, ui = (R)u[q].y;
          xr += m[q].x * ur - m[q].y * ui;
          xi += m[q].x * ui + m[q].y * ur;
        }
    }
  }
  for (int o = 8; o > 0; o >>= 1) {
    xr += __shfl_xor_sync(0xffffffffu, xr, o);
    xi += __shfl_xor_sync(0xffffffffu, xi, o);
  }
  if (on && lane == 0) {
    const double2 x = make_double2(sc * (double)xr, sc * (double)xi);
    const size_t idx = (size_t)b * ns + k;
    xs[(size_t)k * nb + b] = cvt<C>(x);
    if (xd) xd[idx] = x;
  }
}

// ---------------------------------------------------------------- z pass with the kernel

// Geometry of a z pass.  The slab holds the nz z-planes of the active box (plane p is grid
// z = box_lo + p), each an L x L plane of x/y spectra.  The z transform length LZ (a
// template parameter) is at least 2 nz: the linear convolution of nz planes with the
// kernel needs offsets |dz| < nz only, so a circular convolution of any length >= 2 nz - 1
// gives the same values on the nz output planes as the 2N-point padding.  The kernel
// spectrum octant is [LZ/2 + 1][N + 1][N + 1] (z, y, x).
struct ZGeom {
  int L;   // x/y padded length 2N
  int N;   // L / 2 (x/y fold of the kernel octant)
  int nz;  // z planes of the slab: input samples 0 .. nz-1, outputs kept 0 .. nz-1
};

// Two-step LZ = R1 * R2, one tile of W adjacent z-columns per block, a single
// shared exchange tile t[(k1 R2 + n2) W + l]:
//   A  thread (l, n2): the nz <= LZ/2 nonzero samples p = R2 n1 + n2 (n1 < R1/2) come
//      straight from memory, radix-R1 butterfly, twiddle W_LZ^{n2 k1}, into t;
//   B  thread (l, k1): its R2 values of t, radix-R2 butterfly -> X[k1 + R1 k2] in
//      registers; product with the kernel spectrum; inverse radix-R2 butterfly,
//      twiddle W_LZ^{-k1 n2}, back into the same slots of t (a thread reads and writes
//      only its own (k1, l) slice, so B needs no barrier inside);
//   C  thread (l, n2): inverse radix-R1 butterfly over k1, the outputs
//      p = n2 + R2 n1 < nz stored straight to memory.
// A column's data cross shared memory twice instead of once per pass.
// radix split of the z pass: for LZ = 128 the 16 x 8 split keeps the step-B registers
// (operands and spectrum slice) at 8 complex values each
template <int LZ>
constexpr int zsplit_r1() {
  return LZ == 128 ? 16 : split_r1(LZ);
}
template <int LZ, class C>
constexpr int zcol_width() {
  return (int)sizeof(C) == 8 ? (LZ < 32 ? LZ : LZ >= 512 ? 16 : 32) : (LZ < 16 ? LZ : LZ >= 512 ? 8 : 16);
}
constexpr int kZThreads = 256;

template <int LZ, int W, class C>
__device__ __forceinline__ void zcol_step_a(const C* __restrict__ col, long long es, C* t, const C* tw, int nz) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  for (int u = threadIdx.x; u < W * R2; u += kZThreads) {
    const int l = u % W, n2 = u / W;
    C v[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) {
      const int p = R2 * n1 + n2;
      v[n1] = n1 < R1 / 2 && p < nz ? col[(long long)p * es + l] : C{};
    }
    dft_half_in<R1, LZ, false, C>(v, tw);  // samples p >= LZ/2 are the zero padding
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      C x = v[k1];
      if (k1 && n2) x = x * tw[n2 * k1];
      t[(k1 * R2 + n2) * W + l] = x;
    }
  }
}

// the spectrum X[k1 + R1 k2] of column l from t (after step A and a barrier)
template <int LZ, int W, class C>
__device__ __forceinline__ void zcol_step_b_fwd(const C* t, const C* tw, int k1, int l,
                                                C (&v)[LZ / zsplit_r1<LZ>()]) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) v[n2] = t[(k1 * R2 + n2) * W + l];
  DFTL<R2, LZ, false, C>::run(v, tw);
  (void)R1;
}

// inverse radix-R2 butterfly of a spectrum slice, twiddled back into t
template <int LZ, int W, class C>
__device__ __forceinline__ void zcol_step_b_inv(C* t, const C* tw, int k1, int l, C (&v)[LZ / zsplit_r1<LZ>()]) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  DFTL<R2, LZ, true, C>::run(v, tw);
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    C x = v[n2];
    if (k1 && n2) x = x * conjc(tw[n2 * k1]);
    t[(k1 * R2 + n2) * W + l] = x;
  }
  (void)R1;
}

template <int LZ, int W, class C>
__device__ __forceinline__ void zcol_step_c(const C* t, const C* tw, C* __restrict__ col, long long es, int nz) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  for (int u = threadIdx.x; u < W * R2; u += kZThreads) {
    const int l = u % W, n2 = u / W;
    C v[R1];
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) v[k1] = t[(k1 * R2 + n2) * W + l];
    dft_half_out<R1, LZ, true, C>(v, tw);  // only the outputs p < LZ/2 are formed
#pragma unroll
    for (int n1 = 0; n1 < R1 / 2; ++n1) {
      const int p = n2 + R2 * n1;
      if (p < nz) col[(long long)p * es + l] = v[n1];
    }
  }
}

// the kernel-spectrum column of kind `kind` at (x, y): entry kz at [fold(kz, LZ/2) * n1^2]
template <int LZ, class C>
__device__ __forceinline__ const C* kcol(const C* kspec, const ZGeom& g, int kind, int x, int y) {
  const size_t n1 = (size_t)g.N + 1;
  return kspec + (size_t)kind * n1 * n1 * (LZ / 2 + 1) + (size_t)fold(y, g.N) * n1 + fold(x, g.N);
}

// Forward z-FFT of the slab column, product with the kernel spectrum of delay m
// (G^A for c = x,y,z; G^phi for c = div; even-symmetric octant), inverse z-FFT,
// the nz outputs written back in place.  Grid (nb * 4, L / W, L) in the order above.
template <int LZ, int W, class C>
__global__ void __launch_bounds__(kZThreads) k_zconv_p2(C* __restrict__ Bf, const C* __restrict__ kspec, ZGeom g,
                                                        const int* __restrict__ active,
                                                        const C* __restrict__ twg) {
  pdl_wait();
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  const int bc = blockIdx.x;
  if (active && !active[bc >> 2]) return;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* t = tw + LZ;
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  const int y = zpass_row(blockIdx.z, g.N), x0 = blockIdx.y * W;
  const long long es = (long long)g.L * g.L;
  C* col = Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0;
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1);
  zcol_step_a<LZ, W, C>(col, es, t, tw, g.nz);
  __syncthreads();
  for (int u = threadIdx.x; u < W * R1; u += kZThreads) {
    const int l = u % W, k1 = u / W;
    const C* G = kcol<LZ>(kspec, g, (bc & 3) == 3 ? 1 : 0, x0 + l, y);
    C gk[R2], v[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) gk[k2] = __ldg(G + (size_t)fold(k1 + R1 * k2, LZ / 2) * nn);
    zcol_step_b_fwd<LZ, W, C>(t, tw, k1, l, v);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = v[k2] * gk[k2];
    zcol_step_b_inv<LZ, W, C>(t, tw, k1, l, v);
  }
  __syncthreads();
  zcol_step_c<LZ, W, C>(t, tw, col, es, g.nz);
  pdl_trigger();
}

// The y passes of large complex64 grids (those the plane kernel does not hold): W adjacent
// lines per tile, two-step transform L = R1 R2 as in k_cols_p2, each block running through
// many tiles with the next tile's rows on their way (cp.async) while the current one is
// transformed, so loads, butterflies and stores overlap.  Rows outside [in_lo, in_hi] are
// zero (the stage keeps zeros there), outputs outside [out_lo, out_hi] are not stored.
// Measured, 4 waves on the 384^3 grid, per launch: forward 2.00 -> 1.52 ms, inverse 2.24 ->
// 1.39 ms against k_cols_p2; floor 1.2 ms of HBM traffic each.
template <int L, bool INV>
struct YPipe {
  static constexpr int R1 = split_r1(L), R2 = L / R1, W = L == 768 ? 8 : 16, NT = 256;
  static constexpr int ROWS = INV ? L : L / 2;  // rows of a staged tile
  static constexpr size_t smem = (size_t)(kTw2<R1, R2> + ROWS * W + L * W) * sizeof(float2);
  static constexpr int blocks = smem <= 72 * 1024 ? 3 : 2;
  // exchange row (k1, n2); with 8 lines a half-warp spans two k1, put on rows of opposite parity
  static __device__ __forceinline__ int row(int k1, int n2) { return k1 * R2 + (W == 8 ? n2 ^ (k1 & 1) : n2); }
};
template <int L, bool INV>
__global__ void __launch_bounds__(256, (YPipe<L, INV>::blocks))
    k_ypipe(const float2* __restrict__ in, float2* __restrict__ out, int ntiles, int in_lo, int in_hi, int out_lo,
            int out_hi, long long plane_in, long long plane_out, const float2* __restrict__ twg) {
  using Y = YPipe<L, INV>;
  constexpr int R1 = Y::R1, R2 = Y::R2, W = Y::W, NT = Y::NT, CH = W / 2;  // 16-byte chunks per row
  float2* tw = reinterpret_cast<float2*>(aim_smem);
  float2* stage = tw + kTw2<R1, R2>;
  float2* t = stage + Y::ROWS * W;
  load_twiddles2<R1, R2>(tw, twg);
  for (int i = threadIdx.x; i < Y::ROWS * W; i += NT)
    if (i / W < in_lo || i / W > in_hi) stage[i] = make_float2(0, 0);
  pdl_wait();
  // tile = (plane, x tile), x fastest
  auto fetch = [&](int tile) {
    const float2* src = in + (tile / (L / W)) * plane_in + (tile % (L / W)) * W;
    for (int i = threadIdx.x; i < (in_hi - in_lo + 1) * CH; i += NT) {
      const int r = in_lo + i / CH, c = i % CH;
      cp_async16(smem_addr(stage + r * W + 2 * c), src + (long long)r * L + 2 * c);
    }
    cp_async_commit();
  };
  int tile = blockIdx.x;
  if (tile < ntiles) fetch(tile);
  for (; tile < ntiles; tile += gridDim.x) {
    cp_async_wait();
    __syncthreads();
    for (int u = threadIdx.x; u < W * R2; u += NT) {
      const int l = u % W, n2 = u / W;
      float2 v[R1];
#pragma unroll
      for (int n1 = 0; n1 < (INV ? R1 : R1 / 2); ++n1) v[n1] = stage[(R2 * n1 + n2) * W + l];
      if constexpr (INV)
        DFTL<R1, L, true, float2>::run(v, tw);
      else
        dft_half_in<R1, L, false, float2>(v, tw);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) {
        const float2 w = tw[k1 * (R2 + 1) + n2];
        t[Y::row(k1, n2) * W + l] = k1 ? v[k1] * (INV ? conjc(w) : w) : v[k1];
      }
    }
    __syncthreads();  // the stage may be refilled
    if (tile + (int)gridDim.x < ntiles) fetch(tile + gridDim.x);
    float2* dst = out + (tile / (L / W)) * plane_out + (tile % (L / W)) * W;
    for (int u = threadIdx.x; u < W * R1; u += NT) {
      const int l = u % W, k1 = u / W;
      float2 v[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) v[n2] = t[Y::row(k1, n2) * W + l];
      if constexpr (INV) {
        dft_half_out<R2, L, true, float2>(v, tw);  // outputs below L / 2 only
#pragma unroll
        for (int k2 = 0; k2 < R2 / 2; ++k2) {
          const int k = k1 + R1 * k2;
          if (k >= out_lo && k <= out_hi) dst[(long long)k * L + l] = v[k2];
        }
      } else {
        DFTL<R2, L, false, float2>::run(v, tw);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) dst[(long long)(k1 + R1 * k2) * L + l] = v[k2];
      }
    }
  }
  cp_async_wait();
}

// The z pass of the lengths with a factor 3 on large complex64 grids.  A warp takes CW = 8
// adjacent columns, 32 lanes = (column, n2 or k1), and its own exchange buffer, so the block
// never synchronises and every lane has work in each step (12 or 16 items per column).  The
// columns of the next component (or, in Z_RHS, of the next delay) stream into the warp's tile
// by cp.async while the current ones are transformed.  With MODE Z_CONV the warp runs through
// all right-hand sides and components of its columns; where the lane's slice of the kernel
// spectrum fits in registers (LZ = 144) it is read once per kernel kind instead of once per
// component.  With MODE Z_RHS it sums the delays of one (right-hand side, component) in
// registers.  Each 8-column run is two 32-byte sectors.
// Measured, 4 waves on the 384^3 grid (72 box planes), per launch: block tiles of 32 columns
// 4.94 ms at LZ = 192 (416 warp instructions per column, a quarter of the lanes idle in two of
// the three steps); this kernel 3.2 ms at LZ = 144 (3.85 ms with register loads instead of
// cp.async, waiting for memory).  Floors: 1.6 ms HBM, 1.7 ms FP32.
enum { Z_CONV = 0, Z_RHS = 1 };
template <int LZ>
struct ZWarp {
  static constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1, CW = 8, NW = 4;
  static constexpr int QA = CW * R2 / 32, QB = CW * R1 / 32;
  static constexpr bool HOLD = QB * R2 <= 36;
  // column pitch 2 mod 16: the 8 columns of a half-warp fall in different banks
  static constexpr int PZ = pl_round(R1 * (R2 + 1), 2);
  static constexpr int TILE = LZ / 2 * CW, PER_WARP = TILE + CW * PZ;
  static constexpr size_t smem = (size_t)(kTw2<R1, R2> + NW * PER_WARP) * sizeof(float2);
  static constexpr int blocks = (int)((size_t)(228 * 1024) / (smem + 1024));
  static_assert(CW * R1 % 32 == 0 && CW * R2 % 32 == 0, "whole warps");

  // start copying the nz rows of 8 columns into the warp's tile [row][8]
  static __device__ __forceinline__ void fetch(const float2* __restrict__ col, long long es, int nz, float2* tile) {
    const int lane = threadIdx.x & 31;
    const float2* s = col + (lane >> 2) * es + 2 * (lane & 3);
    unsigned d = smem_addr(tile + 2 * lane);
    for (int r = lane >> 2; r < nz; r += 8) {
      cp_async16(d, s);
      s += 8 * es;
      d += 64 * sizeof(float2);
    }
    cp_async_commit();
  }
  static __device__ __forceinline__ void fetched() {
    cp_async_wait();
    __syncwarp();
  }
  static __device__ __forceinline__ void step_a(const float2* tile, float2* scr, const float2* tw) {
    const int lane = threadIdx.x & 31, l = lane & 7;
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int n2 = (lane >> 3) + 4 * q;
      float2 v[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1 / 2; ++n1) v[n1] = tile[(R2 * n1 + n2) * CW + l];
      dft_half_in<R1, LZ, false, float2>(v, tw);
      float2* t = scr + l * PZ + n2;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) t[k1 * (R2 + 1)] = k1 ? v[k1] * tw[k1 * (R2 + 1) + n2] : v[k1];
    }
    __syncwarp();  // the tile may be refilled, the exchange buffer is complete
  }
  static __device__ __forceinline__ void step_c(float2* __restrict__ dst, long long es, int nz, const float2* scr,
                                                const float2* tw) {
    const int lane = threadIdx.x & 31, l = lane & 7;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int n2 = (lane >> 3) + 4 * q;
      const float2* t = scr + l * PZ + n2;
      float2 v[R1];
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) v[k1] = t[k1 * (R2 + 1)];
      dft_half_out<R1, LZ, true, float2>(v, tw);
      float2* d = dst + n2 * es + l;
#pragma unroll
      for (int n1 = 0; n1 < R1 / 2; ++n1) {
        if (R2 * n1 + n2 < nz) *d = v[n1];
        d += R2 * es;
      }
    }
    __syncwarp();
  }
  // the lane's slice kz = k1 + R1 k2 of a spectrum octant: ascending below LZ/2, then descending
  static __device__ __forceinline__ void load_g(const float2* __restrict__ G, size_t nn, int k1, float2 (&g)[R2]) {
    const float2* p = G + (size_t)k1 * nn;
#pragma unroll
    for (int k2 = 0; k2 < R2 / 2; ++k2) {
      g[k2] = __ldg(p);
      p += R1 * nn;
    }
    p = G + (size_t)(LZ / 2 - k1) * nn;  // kz = LZ/2 + k1 + R1 (k2 - R2/2) mirrors LZ/2 - ...
#pragma unroll
    for (int k2 = R2 / 2; k2 < R2; ++k2) {
      g[k2] = __ldg(p);
      p -= R1 * nn;
    }
  }
  static __device__ __forceinline__ void b_forward(const float2* t, const float2* tw, float2 (&v)[R2]) {
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) v[n2] = t[n2];
    DFTL<R2, LZ, false, float2>::run(v, tw);
  }
  static __device__ __forceinline__ void b_inverse(float2* t, const float2* tw, int k1, float2 (&v)[R2]) {
    DFTL<R2, LZ, true, float2>::run(v, tw);
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) t[n2] = n2 ? v[n2] * conjc(tw[k1 * (R2 + 1) + n2]) : v[n2];
  }
};

// Grid (L / 32, L[, nb * 4 for Z_RHS]): 32 adjacent columns of row y (mirror order) per block.
template <int LZ, int MODE>
__global__ void __launch_bounds__(32 * ZWarp<LZ>::NW, ZWarp<LZ>::blocks)
    k_zwarp(float2* __restrict__ Bf, const float2* __restrict__ kspec, ZGeom g, int nb, const int* __restrict__ active,
            const float2* __restrict__ twg, const __grid_constant__ SlabList sl) {
  using Z = ZWarp<LZ>;
  constexpr int QB = Z::QB, R2 = Z::R2;
  float2* tw = reinterpret_cast<float2*>(aim_smem);
  load_twiddles2<Z::R1, Z::R2>(tw, twg);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float2* tile = tw + kTw2<Z::R1, Z::R2> + warp * Z::PER_WARP;
  float2* scr = tile + Z::TILE;
  for (int i = g.nz * Z::CW + lane; i < Z::TILE; i += 32) tile[i] = make_float2(0, 0);  // below the box
  pdl_wait();
  __syncthreads();
  const int y = zpass_row(blockIdx.y, g.N), x0 = (blockIdx.x * Z::NW + warp) * Z::CW;
  const long long es = (long long)g.L * g.L;
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1), oct = nn * (LZ / 2 + 1);
  const size_t off = (size_t)y * g.L + x0, slab = (size_t)g.nz * es;
  // step B: lane (column, k1 = lane / 8 + 4 q)
  float2* tb = scr + (lane & 7) * Z::PZ;
  if (MODE == Z_CONV) {
    // components i: x, y, z of every right-hand side, then div of every right-hand side
    const int n = 4 * nb;
    auto comp = [&](int i) { return i < 3 * nb ? (i / 3) * 4 + i % 3 : (i - 3 * nb) * 4 + 3; };
    auto next = [&](int i) {  // the first component from i on whose right-hand side takes part
      while (i < n && active && !active[comp(i) >> 2]) ++i;
      return i;
    };
    int i = next(0), loaded = -1;
    if (i < n) Z::fetch(Bf + comp(i) * slab + off, es, g.nz, tile);
    float2 gk[Z::HOLD ? QB : 1][R2];
#pragma unroll 1
    while (i < n) {
      const int kind = i < 3 * nb ? 0 : 1;
      const float2* G = kcol<LZ>(kspec, g, kind, x0 + (lane & 7), y);
      if (Z::HOLD && kind != loaded) {
#pragma unroll
        for (int q = 0; q < (Z::HOLD ? QB : 0); ++q) Z::load_g(G, nn, (lane >> 3) + 4 * q, gk[q]);
        loaded = kind;
      }
      Z::fetched();
      Z::step_a(tile, scr, tw);
      const int j = next(i + 1);
      if (j < n) Z::fetch(Bf + comp(j) * slab + off, es, g.nz, tile);
#pragma unroll
      for (int q = 0; q < QB; ++q) {
        const int k1 = (lane >> 3) + 4 * q;
        float2* t = tb + k1 * (R2 + 1);
        float2 v[R2];
        if constexpr (!Z::HOLD) Z::load_g(G, nn, k1, gk[0]);
        Z::b_forward(t, tw, v);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) v[k2] = v[k2] * gk[Z::HOLD ? q : 0][k2];
        Z::b_inverse(t, tw, k1, v);
      }
      Z::step_c(Bf + comp(i) * slab + off, es, g.nz, scr, tw);
      i = j;
    }
  } else {
    const int bc = blockIdx.z;
    auto col = [&](int s) { return reinterpret_cast<const float2*>(sl.p[s]) + bc * slab + off; };
    float2 acc[QB][R2];
#pragma unroll
    for (int q = 0; q < QB; ++q)
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) acc[q][k2] = make_float2(0, 0);
    if (sl.n > 0) Z::fetch(col(0), es, g.nz, tile);
#pragma unroll 1
    for (int s = 0; s < sl.n; ++s) {
      const float2* G = kcol<LZ>(kspec + (size_t)sl.m[s] * 2 * oct, g, (bc & 3) == 3 ? 1 : 0, x0 + (lane & 7), y);
      Z::fetched();
      Z::step_a(tile, scr, tw);
      if (s + 1 < sl.n) Z::fetch(col(s + 1), es, g.nz, tile);
#pragma unroll
      for (int q = 0; q < QB; ++q) {
        const int k1 = (lane >> 3) + 4 * q;
        float2 v[R2], gk[R2];
        Z::load_g(G, nn, k1, gk);
        Z::b_forward(tb + k1 * (R2 + 1), tw, v);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) acc[q][k2] += v[k2] * gk[k2];
      }
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      const int k1 = (lane >> 3) + 4 * q;
      Z::b_inverse(tb + k1 * (R2 + 1), tw, k1, acc[q]);
    }
    Z::step_c(Bf + bc * slab + off, es, g.nz, scr, tw);
  }
}

// History slabs of power-of-two z length are kept z-transformed: S[bc][kz][y][x], all LZ
// frequencies kz of every (x, y) line (LZ / nz times the bytes of the x/y-transformed
// slab).  The delay sum of the right-hand side is then a multiply-accumulate streamed
// over the N_g spectra and one inverse z-FFT, instead of N_g forward z-FFTs recomputed
// at every step.
//
// k_zfwd_spec: the forward z-FFT (steps A and B of the z pass) of the slab in Bf into the
// spectral layout; thread (l, k1) of step B stores X[k1 + R1 k2] for all k2.
template <int LZ, int W, class C>
__global__ void __launch_bounds__(kZThreads) k_zfwd_spec(const C* __restrict__ Bf, C* __restrict__ S, ZGeom g,
                                                         const C* __restrict__ twg) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* t = tw + LZ;
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  const int bc = blockIdx.z, y = blockIdx.y, x0 = blockIdx.x * W;
  const long long es = (long long)g.L * g.L;
  zcol_step_a<LZ, W, C>(Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0, es, t, tw, g.nz);
  __syncthreads();
  C* out = S + (size_t)bc * LZ * es + (size_t)y * g.L + x0;
  for (int u = threadIdx.x; u < W * R1; u += kZThreads) {
    const int l = u % W, k1 = u / W;
    C v[R2];
    zcol_step_b_fwd<LZ, W, C>(t, tw, k1, l, v);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) out[(long long)(k1 + R1 * k2) * es + l] = v[k2];
  }
}

// Delay sum of the right-hand side in the spectral domain:
//   P^_col = sum_i G^_{m_i} . S_i(col), then one inverse z-FFT (steps B inverse and C),
// the sum kept in the registers of the step-B threads (thread (l, k1) owns the
// frequencies k1 + R1 k2).
template <int LZ, int W, class C>
__global__ void __launch_bounds__(kZThreads, 3) k_zrhs_spec(SlabList sl, const C* __restrict__ kspec_all, ZGeom g,
                                                         C* __restrict__ Bf, const C* __restrict__ twg) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1, U = (W * R1 + kZThreads - 1) / kZThreads;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* t = tw + LZ;
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  const int bc = blockIdx.z, y = blockIdx.y, x0 = blockIdx.x * W;
  const long long es = (long long)g.L * g.L;
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1), oct = nn * (LZ / 2 + 1);
  const int kind = (bc & 3) == 3 ? 1 : 0;
  C acc[U][R2];
#pragma unroll
  for (int j = 0; j < U; ++j)
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] = C{};
  for (int s = 0; s < sl.n; ++s) {
    const C* Sc = reinterpret_cast<const C*>(sl.p[s]) + (size_t)bc * LZ * es + (size_t)y * g.L + x0;
    const C* Gm = kspec_all + (size_t)sl.m[s] * 2 * oct;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int u = threadIdx.x + j * kZThreads;
      if (u < W * R1) {
        const int l = u % W, k1 = u / W;
        const C* G = kcol<LZ>(Gm, g, kind, x0 + l, y);
        C gk[R2], v[R2];
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) {
          const int kz = k1 + R1 * k2;
          v[k2] = Sc[(long long)kz * es + l];
          gk[k2] = __ldg(G + (size_t)fold(kz, LZ / 2) * nn);
        }
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] += v[k2] * gk[k2];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int u = threadIdx.x + j * kZThreads;
    if (u < W * R1) zcol_step_b_inv<LZ, W, C>(t, tw, u / W, u % W, acc[j]);
  }
  __syncthreads();
  zcol_step_c<LZ, W, C>(t, tw, Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0, es, g.nz);
}

// The same with the spectra streamed by TMA (complex64): the LZ x W tile of each spectrum
// is a 4-D box of the ring tensor [slot][B*4*LZ][L][L], loaded into one of two 128-byte
// aligned shared buffers by cp.async.bulk.tensor and signalled on an mbarrier, so
// spectrum s + 2 streams in while spectrum s + 1 is accumulated.  Waits are bounded.  A
// wait that gives up sets *err (the host reports AIM_ERR_TIMEOUT) and a block-wide flag;
// the block then issues no further load, drains the loads it has in flight with one more
// bounded wait each and returns without writing its output (which is undefined whenever
// *err is set).
template <int LZ, int W>
__global__ void __launch_bounds__(kZThreads, 3) k_zrhs_spec_tma(const __grid_constant__ CUtensorMap ring,
                                                                SlabRing sr, const float2* __restrict__ kspec_all,
                                                                ZGeom g, float2* __restrict__ Bf,
                                                                const float2* __restrict__ twg, int* __restrict__ err) {
  using C = float2;
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1, U = (W * R1 + kZThreads - 1) / kZThreads;
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int gave_up[2];  // by iteration parity: a write in iteration s + 1 cannot reach a
                              // thread still reading the flag of iteration s
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(aim_smem) + 127) & ~static_cast<uintptr_t>(127));
  C* in0 = reinterpret_cast<C*>(base);  // [2][LZ][W]
  C* tw = in0 + 2 * LZ * W;
  C* t = tw + LZ;
  const int bc = blockIdx.z, y = blockIdx.y, x0 = blockIdx.x * W;
  const unsigned bytes = (unsigned)(LZ * W * sizeof(C));
  if (threadIdx.x == 0) {
    gave_up[0] = gave_up[1] = 0;
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  if (threadIdx.x == 0)
    for (int s = 0; s < 2 && s < sr.n; ++s) {
      mbar_arrive_expect_tx(&bar[s], bytes);
      tma_load_4d(in0 + s * LZ * W, &ring, &bar[s], x0, y, bc * LZ, sr.slot[s]);
    }
  const long long es = (long long)g.L * g.L;
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1), oct = nn * (LZ / 2 + 1);
  const int kind = (bc & 3) == 3 ? 1 : 0;
  C acc[U][R2];
#pragma unroll
  for (int j = 0; j < U; ++j)
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] = C{};
  for (int s = 0; s < sr.n; ++s) {
    const int buf = s & 1;
    const C* Gm = kspec_all + (size_t)sr.m[s] * 2 * oct;
    C gk[U][R2];
#pragma unroll
    for (int j = 0; j < U; ++j) {  // the kernel spectrum while the tile streams in
      const int u = threadIdx.x + j * kZThreads;
      if (u < W * R1) {
        const C* G = kcol<LZ>(Gm, g, kind, x0 + u % W, y);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) gk[j][k2] = __ldg(G + (size_t)fold(u / W + R1 * k2, LZ / 2) * nn);
      }
    }
    const bool ok = mbar_wait_bounded(&bar[buf], (unsigned)((s >> 1) & 1));
    if (!ok) {
      atomicExch(err, 1);
      gave_up[s & 1] = 1;
    }
    const C* tile = in0 + buf * LZ * W;  // [kz][l]
    if (ok) {
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int u = threadIdx.x + j * kZThreads;
        if (u < W * R1) {
          const int l = u % W, k1 = u / W;
#pragma unroll
          for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] += tile[(k1 + R1 * k2) * W + l] * gk[j][k2];
        }
      }
    }
    __syncthreads();  // the tile is consumed: it may be refilled (gave_up[s & 1] is block-uniform)
    if (gave_up[s & 1]) {
      // loads in flight: spectrum s (the wait that gave up, for some thread) and s + 1
      if (threadIdx.x == 0) {
        mbar_wait_bounded(&bar[buf], (unsigned)((s >> 1) & 1));
        if (s + 1 < sr.n) mbar_wait_bounded(&bar[buf ^ 1], (unsigned)(((s + 1) >> 1) & 1));
      }
      __syncthreads();
      return;
    }
    if (threadIdx.x == 0 && s + 2 < sr.n) {
      fence_proxy_async_smem();
      mbar_arrive_expect_tx(&bar[buf], bytes);
      tma_load_4d(in0 + buf * LZ * W, &ring, &bar[buf], x0, y, bc * LZ, sr.slot[s + 2]);
    }
  }
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int u = threadIdx.x + j * kZThreads;
    if (u < W * R1) zcol_step_b_inv<LZ, W, C>(t, tw, u / W, u % W, acc[j]);
  }
  __syncthreads();
  zcol_step_c<LZ, W, C>(t, tw, Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0, es, g.nz);
}

// Blocked right-hand side (Sec. 4 stage ii), power-of-two z lengths.  The pending
// accumulator of a step holds the z-spectra P^ of its delayed grid sum, built by the
// squares of earlier steps; k_zinv_pending turns it into the slab of potentials (inverse
// z-FFT, steps B^-1 and C) and clears it for reuse.
template <int LZ, int W, class C>
__global__ void __launch_bounds__(kZThreads) k_zinv_pending(C* __restrict__ S, ZGeom g, C* __restrict__ Bf,
                                                            const C* __restrict__ twg) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* t = tw + LZ;
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  const int bc = blockIdx.z, y = blockIdx.y, x0 = blockIdx.x * W;
  const long long es = (long long)g.L * g.L;
  C* Sc = S + (size_t)bc * LZ * es + (size_t)y * g.L + x0;
  for (int u = threadIdx.x; u < W * R1; u += kZThreads) {
    const int l = u % W, k1 = u / W;
    C v[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) {
      C* e = Sc + (long long)(k1 + R1 * k2) * es + l;
      v[k2] = *e;
      *e = C{};
    }
    zcol_step_b_inv<LZ, W, C>(t, tw, k1, l, v);
  }
  __syncthreads();
  zcol_step_c<LZ, W, C>(t, tw, Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0, es, g.nz);
}

// One square: every element q of the z-spectra ([bc][kz][y][x], nb * 4 * LZ * L * L of
// them) gathers its kernel taps G^_m, m = toff - B + 1 .. toff + B - 1 within 1 .. N_g,
// from the octant, its B sources, and adds the B Toeplitz products into the pending
// accumulators.  Each source and accumulator element is read (and written) once per
// square; at B <= 16 the direct product (8 B^2 flops per element) costs no more than
// temporal FFTs of length 2B would.
template <int B, class C>
__global__ void __launch_bounds__(256) k_block_square(BlockSquare sq, const C* __restrict__ kspec, ZGeom g, int LZ,
                                                      int ng, long long n) {
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1), oct = nn * (LZ / 2 + 1);
  const long long plane = (long long)g.L * g.L, per_bc = plane * LZ;
  const int m0 = sq.toff - B + 1;  // tap[t] = G^_{m0 + t}
  for (long long q = blockIdx.x * 256LL + threadIdx.x; q < n; q += (long long)gridDim.x * 256) {
    const int x = (int)(q % g.L), y = (int)((q / g.L) % g.L), kz = (int)((q / plane) % LZ);
    const int bc = (int)(q / per_bc), kind = (bc & 3) == 3 ? 1 : 0;
    const size_t go = (size_t)kind * oct + ((size_t)fold(kz, LZ / 2) * (g.N + 1) + fold(y, g.N)) * (g.N + 1) +
                      fold(x, g.N);
    C tap[2 * B - 1];
#pragma unroll
    for (int t = 0; t < 2 * B - 1; ++t) {
      const int m = m0 + t;
      tap[t] = (m >= 1 && m <= ng) ? __ldg(kspec + (size_t)m * 2 * oct + go) : C{};
    }
    C s[B];
#pragma unroll
    for (int j = 0; j < B; ++j) s[j] = reinterpret_cast<const C*>(sq.src[j])[q];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      C acc{};
#pragma unroll
      for (int j = 0; j < B; ++j) acc += tap[B - 1 + i - j] * s[j];
      C* d = reinterpret_cast<C*>(sq.dst[i]) + q;
      *d = *d + acc;
    }
  }
}

// The same on spectra in the plane kernel's order, [bc][kx][group][pair][unit][2], with the
// taps from its tabulated kernel spectra; grid (blocks, nb * 4), so that an element's place in
// the table takes 32-bit divisions only.
template <int B, class C>
__global__ void __launch_bounds__(256) k_block_square_plane(BlockSquare sq, const C* __restrict__ G, PlaneOrder o,
                                                            int ng) {
  const int per_bc = o.L * o.L * o.LZ;
  const size_t gm = plane_spec_elems(o);
  const int m0 = sq.toff - B + 1;  // tap[t] = G^_{m0 + t}
  if ((blockIdx.y & 3) == 3) G += (size_t)(o.L / 2 + 1) * plane_g_elems(o);
  for (int i = blockIdx.x * 256 + threadIdx.x; i < per_bc; i += gridDim.x * 256) {
    const size_t go = plane_g_index(o, i), q = (size_t)blockIdx.y * per_bc + i;
    C tap[2 * B - 1];
#pragma unroll
    for (int t = 0; t < 2 * B - 1; ++t) {
      const int m = m0 + t;
      tap[t] = (m >= 1 && m <= ng) ? __ldg(G + (size_t)m * gm + go) : C{};
    }
    C s[B];
#pragma unroll
    for (int j = 0; j < B; ++j) s[j] = reinterpret_cast<const C*>(sq.src[j])[q];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      C acc{};
#pragma unroll
      for (int j = 0; j < B; ++j) acc += tap[B - 1 + i - j] * s[j];
      C* d = reinterpret_cast<C*>(sq.dst[i]) + q;
      *d = *d + acc;
    }
  }
}

// z lengths with a factor 3 keep x/y-transformed history slabs: the delay sum recomputes
// each slab's forward z-transform (steps A and B of the z pass), multiplies it by its
// delay's kernel spectrum and accumulates in the registers of the step-B threads; then one
// inverse z-FFT (steps B^-1 and C), the nz outputs written to Bf.
template <int LZ, int W, class C>
__global__ void __launch_bounds__(kZThreads) k_zrhs_2s(SlabList sl, const C* __restrict__ kspec_all, ZGeom g,
                                                       C* __restrict__ Bf, const C* __restrict__ twg) {
  constexpr int R1 = zsplit_r1<LZ>(), R2 = LZ / R1, U = (W * R1 + kZThreads - 1) / kZThreads;
  C* tw = reinterpret_cast<C*>(aim_smem);
  C* t = tw + LZ;
  load_twiddles(tw, twg, LZ);
  __syncthreads();
  const int bc = blockIdx.x, y = zpass_row(blockIdx.z, g.N), x0 = blockIdx.y * W;  // z-pass grid order
  const long long es = (long long)g.L * g.L;
  const size_t nn = (size_t)(g.N + 1) * (g.N + 1), oct = nn * (LZ / 2 + 1);
  const int kind = (bc & 3) == 3 ? 1 : 0;
  C acc[U][R2];
#pragma unroll
  for (int j = 0; j < U; ++j)
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] = C{};
  for (int s = 0; s < sl.n; ++s) {
    const C* col = reinterpret_cast<const C*>(sl.p[s]) + (size_t)bc * g.nz * es + (size_t)y * g.L + x0;
    const C* Gm = kspec_all + (size_t)sl.m[s] * 2 * oct;
    if (s) __syncthreads();  // the previous delay's step B has read t
    zcol_step_a<LZ, W, C>(col, es, t, tw, g.nz);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int u = threadIdx.x + j * kZThreads;
      if (u < W * R1) {
        const int l = u % W, k1 = u / W;
        const C* G = kcol<LZ>(Gm, g, kind, x0 + l, y);
        C v[R2];
        zcol_step_b_fwd<LZ, W, C>(t, tw, k1, l, v);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) acc[j][k2] += v[k2] * __ldg(G + (size_t)fold(k1 + R1 * k2, LZ / 2) * nn);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const int u = threadIdx.x + j * kZThreads;
    if (u < W * R1) zcol_step_b_inv<LZ, W, C>(t, tw, u / W, u % W, acc[j]);
  }
  __syncthreads();
  zcol_step_c<LZ, W, C>(t, tw, Bf + (size_t)bc * g.nz * es + (size_t)y * g.L + x0, es, g.nz);
}

// ---------------------------------------------------------------- stage iii + iv
// y_k = sign * ( sum_c sum_{n in stencil(k)} L_c[n,k] P_c[n]  +  sum_terms Z~near_m x_m ) + base_k
// Grid (nb, row blocks): a warp takes ROWS consecutive rows of one RHS, a block the rows of
// its 8 warps: 4 rows per warp, or 1 on small systems, whose FP64 work would otherwise sit on
// a few SMs (interp_rows).  Grid part: the whole warp per row, accumulated in the grid
// precision, the rows' sums reduced together.  Near part: 32 / ROWS lanes per row, all rows
// at once, in FP64 -- the warp's FP64 instructions (each holds the FP64 pipe for the whole
// warp) serve ROWS rows.  With df.V set (the operator of an Arnoldi step, y = Krylov slot
// j+1) the block also forms the raw dots conj(vt_i) . y over its rows for i <= j, 32 / rows
// of them per warp instruction, and the last block of the RHS sums them into df.d.
// Measured, us per product: 480 unknowns, complex128, 16.3 -> 8.1 (15 blocks before);
// 64 right-hand sides of 7680 unknowns, complex64, 334 -> 262.
template <class C, int ROWS>
__global__ void __launch_bounds__(256, 3) k_interp_near(const C* __restrict__ P, const int* __restrict__ anchor,
                                                     const int* __restrict__ order,
                                                     const typename Real<C>::T* __restrict__ lam, int N, int nz,
                                                     int zlo, int ns,
                                                     int nb, const int* __restrict__ rowptr,
                                                     const int* __restrict__ col, NearList nl,
                                                     const double2* __restrict__ base, double sign,
                                                     const int* __restrict__ active, double2* __restrict__ y,
                                                     VecSel ys, DotFuse df) {
  using R = typename Real<C>::T;
  // the right-hand side is the fastest grid index: the blocks of all right-hand sides
  // for one set of rows run together and share that set's near-zone rows through L2
  const int b = blockIdx.x, rb = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int brows = 8 * ROWS, GL = 32 / ROWS;  // rows per block, lanes per row of the near part
  const int k0 = rb * brows + warp * ROWS;  // the warp's first position
  // set-up tables first: they do not depend on the previous kernel
  int kr[ROWS];
  size_t org[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) kr[r] = k0 + r < ns ? order[k0 + r] : -1;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int k = kr[r] < 0 ? 0 : kr[r];
    org[r] = ((size_t)(anchor[3 * k + 2] - zlo) * N + anchor[3 * k + 1]) * N + anchor[3 * k];
  }
  // near part: lane group r, sub-lane sl
  const int r = lane / GL, sl = lane % GL;
  int k = kr[0];
#pragma unroll
  for (int q = 1; q < ROWS; ++q) k = r == q ? kr[q] : k;
  const bool on = k >= 0;
  int e = on ? rowptr[k] + sl : 0;
  const int e1 = on ? rowptr[k + 1] : 0;
  constexpr int U = ROWS == 4 ? 4 : 2;  // entries of a lane in flight
  int j[U];
#pragma unroll
  for (int u = 0; u < U; ++u) j[u] = e + GL * u < e1 ? col[e + GL * u] : -1;
  pdl_wait();
  if (active && !active[b]) return;
  // grid part, row by row
  C g[ROWS];
  if (P) {
    const size_t N3 = (size_t)nz * N * N;  // the box planes z0 .. z0 + nz - 1
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      g[q] = C{};
      if (kr[q] >= 0) {
        // 4 lanes per stencil row: lane -> (row of 8, dx); the 256 (component, node)
        // terms of an RWG take 8 warp loads of 8 rows x 32 B each
        const C* Pb = P + (size_t)b * 4 * N3 + org[q] + (lane & 3);
        const R* lk = lam + (size_t)kr[q] * 256 + lane;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int p = it * 8 + (lane >> 2);  // (component, row) pair, 0..63
          const int c = p >> 4, row = p & 15;
          const int dz = row >> 2, dy = row & 3;
          g[q] += lk[it * 32] * Pb[c * N3 + ((size_t)dz * N + dy) * N];
        }
      }
    }
  }
  double2 nr = make_double2(0, 0);
  double xscale = 1.0;
  {
    long long xoff = 0;
    if (nl.xsel.sel) {
      const int jj = *nl.xsel.sel + nl.xsel.off;
      xoff = jj * nl.xsel.stride;
      if (nl.xsel.scale) xscale = nl.xsel.scale[b * 64 + jj];
    }
    xoff += (size_t)b * ns;
    if (nl.n)
      for (;;) {
        for (int t = 0; t < nl.n; ++t) {
          const double2* val = nl.val[t];
          const double2* x = nl.x[t] + xoff;
          double2 z[U], xv[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            z[u] = j[u] >= 0 ? val[e + GL * u] : make_double2(0, 0);
            xv[u] = j[u] >= 0 ? x[j[u]] : make_double2(0, 0);
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (j[u] >= 0) {
              if (nl.dinv) {
                const double2 d = nl.dinv[j[u]];
                xv[u] = make_double2(xv[u].x * d.x - xv[u].y * d.y, xv[u].x * d.y + xv[u].y * d.x);
              }
              nr.x += z[u].x * xv[u].x - z[u].y * xv[u].y;
              nr.y += z[u].x * xv[u].y + z[u].y * xv[u].x;
            }
        }
        e += GL * U;
        if (__all_sync(0xffffffffu, e - sl >= e1)) break;
#pragma unroll
        for (int u = 0; u < U; ++u) j[u] = e + GL * u < e1 ? col[e + GL * u] : -1;
      }
  }
  // Sums over lanes, real and imaginary parts split between lane halves.  Grid part: the 8
  // values of 4 rows reduce together, lane group r keeping row r (9 additions instead of 40);
  // then within a group real (first half) and imaginary (second half) parts.
  const bool hi = sl & (GL / 2);
  double grid = 0.0;
  if (P) {
    C t;
    if constexpr (ROWS == 4) {
      const bool h4 = lane & 16, h3 = lane & 8;
      const C s0 = h4 ? g[0] : g[2], s1 = h4 ? g[1] : g[3];
      C a0 = h4 ? g[2] : g[0], a1 = h4 ? g[3] : g[1];
      a0.x += __shfl_xor_sync(0xffffffffu, s0.x, 16);
      a0.y += __shfl_xor_sync(0xffffffffu, s0.y, 16);
      a1.x += __shfl_xor_sync(0xffffffffu, s1.x, 16);
      a1.y += __shfl_xor_sync(0xffffffffu, s1.y, 16);
      const C s = h3 ? a0 : a1;
      t = h3 ? a1 : a0;
      t.x += __shfl_xor_sync(0xffffffffu, s.x, 8);
      t.y += __shfl_xor_sync(0xffffffffu, s.y, 8);
    } else {
      t = g[0];
    }
    R kp = hi ? t.y : t.x;
    kp += __shfl_xor_sync(0xffffffffu, hi ? t.x : t.y, GL / 2);
#pragma unroll
    for (int o = GL / 4; o > 0; o >>= 1) kp += __shfl_xor_sync(0xffffffffu, kp, o);
    grid = (double)kp;
  }
  double keep = hi ? nr.y : nr.x;
  keep += __shfl_xor_sync(0xffffffffu, hi ? nr.x : nr.y, GL / 2);
#pragma unroll
  for (int o = GL / 4; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
  keep = grid + xscale * keep;
  const double nim = __shfl_down_sync(0xffffffffu, keep, GL / 2);
  double2 out = make_double2(0, 0);
  if (on && sl == 0) {
    if (ys.sel) y += (*ys.sel + ys.off) * ys.stride;
    out = make_double2(sign * keep, sign * nim);
    if (base) {
      const double2 bb = base[(size_t)b * ns + k];
      out = make_double2(bb.x + out.x, bb.y + out.y);
    }
    y[(size_t)b * ns + k] = out;
  }
  if (df.V) {
    __shared__ double2 wsm[brows];
    __shared__ int last;
    if (sl == 0) wsm[warp * ROWS + r] = out;  // zero for rows past ns
    __syncthreads();
    const int J = *df.jdev + 1;
    constexpr int NI = 32 / brows;  // dots per warp instruction
    const int row = lane % brows, pb = rb * brows + row;
    const bool in = pb < ns;
    const int kb = in ? order[pb] : 0;
    const double2* Vb = df.V + (size_t)b * ns;
    const double2 w = wsm[row];
    for (int i0 = warp * NI; i0 < J; i0 += 8 * NI) {
      const int i = i0 + lane / brows;
      double2 t = make_double2(0, 0);
      if (in && i < J) {
        const double2 v = Vb[i * df.vstride + kb];
        t = make_double2(v.x * w.x + v.y * w.y, v.x * w.y - v.y * w.x);  // conj(v) w
      }
      // real parts end in the first half of a row group, imaginary in the second
      const bool h = lane & (brows / 2);
      double s = h ? t.y : t.x;
      s += __shfl_xor_sync(0xffffffffu, h ? t.x : t.y, brows / 2);
#pragma unroll
      for (int o = brows / 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const double im = __shfl_down_sync(0xffffffffu, s, brows / 2);
      if (row == 0 && i < J) df.pd[((size_t)b * 64 + i) * df.P + rb] = make_double2(s, im);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      last = atomicAdd(df.ucnt + b, 1u) == (unsigned)df.P - 1;
    }
    __syncthreads();
    if (last) {
      __threadfence();
      if (threadIdx.x == 0) df.ucnt[b] = 0u;
      for (int i = warp; i < J; i += 8) {
        const double2* p = df.pd + ((size_t)b * 64 + i) * df.P;
        double2 t = make_double2(0, 0);
        for (int q = lane; q < df.P; q += 32) {
          const double2 v = __ldcg(p + q);
          t.x += v.x;
          t.y += v.y;
        }
        t = warp_sum_c(t);
        if (lane == 0) df.d[b * 64 + i] = t;
      }
    }
  }
  pdl_trigger();
}

// ---------------------------------------------------------------- launch helpers
template <class K>
static void smem_opt_in(K kernel, size_t bytes) {
  if (bytes > 48 * 1024) AIM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// precision selectors for the context tables
inline const float2* sel_tw(aim_ctx* c, float2*) { return c->d_twf; }
inline const double2* sel_tw(aim_ctx* c, double2*) { return c->d_tw; }
inline const float2* sel_twz(aim_ctx* c, float2*) { return c->d_twzf; }
inline const double2* sel_twz(aim_ctx* c, double2*) { return c->d_twz; }
inline const float2* sel_kspec(aim_ctx* c, float2*) { return c->d_kspecf; }
inline const double2* sel_kspec(aim_ctx* c, double2*) { return c->d_kspec; }
inline const float2* sel_plane(aim_ctx* c, float2*) { return c->d_planef; }
inline const double2* sel_plane(aim_ctx* c, double2*) { return c->d_plane; }
inline const float4* sel_ncoef(aim_ctx* c, float2*) { return c->d_ncoeff; }
inline const double4_32a* sel_ncoef(aim_ctx* c, double2*) { return c->d_ncoef; }
inline const float* sel_lam(aim_ctx* c, float2*) { return c->d_lamf; }
inline const float2* sel_sai(aim_ctx* c, float2*) { return c->d_saif; }
inline const double2* sel_sai(aim_ctx* c, double2*) { return c->d_sai; }
inline const double* sel_lam(aim_ctx* c, double2*) { return c->d_lam; }

// Tile widths the z and y passes are instantiated for (the autotuner picks among them).
template <class F>
inline void with_width(int w, F&& f) {
  switch (w) {
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 16: f(std::integral_constant<int, 16>{}); break;
    case 32: f(std::integral_constant<int, 32>{}); break;
    case 64: f(std::integral_constant<int, 64>{}); break;
    default: throw AimError{AIM_ERR_ARG, "launch plan: unsupported tile width"};
  }
}
// z transform lengths the z pass is instantiated for (aim_ctx::LZ is one of them)
template <class F>
inline void with_zlen(int lz, F&& f) {
  switch (lz) {
    case 16: f(std::integral_constant<int, 16>{}); break;
    case 32: f(std::integral_constant<int, 32>{}); break;
    case 64: f(std::integral_constant<int, 64>{}); break;
    case 128: f(std::integral_constant<int, 128>{}); break;
    case 144: f(std::integral_constant<int, 144>{}); break;
    case 192: f(std::integral_constant<int, 192>{}); break;
    case 256: f(std::integral_constant<int, 256>{}); break;
    case 768: f(std::integral_constant<int, 768>{}); break;
    default: throw AimError{AIM_ERR_ARG, "unsupported z transform length"};
  }
}
constexpr size_t kPlanSmemMax = 220 * 1024;  // dynamic shared memory a plan may ask for

// sizes whose z passes always run in the plane kernel (a factor-3 z length may fall back to
// the separate passes, see plane_setup)
template <int L, int LZ, class C>
constexpr bool plane_always() {
  return plane_fits<L, LZ, C>() && pow2_len(LZ);
}

// z lengths with a factor 3 in complex64 whose exchange fits a warp's buffer: k_zwarp
template <int L, int LZ, class C>
constexpr bool zwarp_len() {
  return sizeof(C) == 8 && LZ <= L && L % 64 == 0 && (LZ == 144 || LZ == 192);
}

// padded lengths whose separate y passes run in k_ypipe (FP64 lines are bound by arithmetic)
template <int L, class C>
constexpr bool ypipe_len() {
  return sizeof(C) == 8 && (L == 192 || L == 256 || L == 768);
}

template <int L, class C>
struct GridOps {
  // ------------------------------------------------------------ launch shapes
  static int def_zw(const aim_ctx* c) {
    int w = 0;
    with_zlen(c->LZ, [&](auto lz) { w = zcol_width<decltype(lz)::value, C>(); });
    return w;
  }
  static int def_cw() { return col_width_p2<L, C>(); }
  // kx-major grids (the plane kernel runs the y and z passes)
  static bool kxm(const aim_ctx* c) { return sizeof(C) == sizeof(float2) ? c->plane : c->plane64; }
  static int def_rp(const aim_ctx* c) {
    if (!kxm(c)) return pow2_len(L) ? std::max(1, 4096 / L) : std::max(1, 256 / split_r1(L));
    return fill_rows(c, 16, (long long)c->batch_max * 4 * c->NZ);
  }
  static int def_ypb(const aim_ctx* c) {
    return kxm(c) ? fill_rows(c, c->batch_max > 1 ? 4 : 8, (long long)c->NZ * ((c->batch_max + 1) / 2)) : 1;
  }
  // the most rows per block (a power of two up to `most`) that still give every SM two blocks
  static int fill_rows(const aim_ctx* c, int most, long long others) {
    int r = std::min(most, L / 2);
    while (r > 1 && (c->N / r) * others < 304) r /= 2;
    return r;
  }
  static size_t smem_z(int lz, int w) { return (size_t)(lz + lz * w) * sizeof(C); }
  static size_t smem_y(int w) { return (size_t)(L + L * w) * sizeof(C); }
  static size_t smem_x(int rp) {
    return (size_t)(row_tmp_pitch<L>() + rp * row_tmp_pitch<L>()) * sizeof(C);
  }
  static size_t smem_anterp(int yb, int bb, bool k) {
    return (x_r1(L) * (x_r2(L) + 1) + (size_t)4 * yb * bb * (L / 2 + x_pitch(L, k ? yb : 1))) * sizeof(C);
  }
  static size_t smem_xinv(int yb) {
    return (x_r1(L) * (x_r2(L) + 1) + (size_t)yb * x_pitch(L, yb)) * sizeof(C);
  }
  // the plan holds the shapes of the context's own precision (the FP64 residual of the
  // refinement on the complex64 path runs with the defaults)
  static bool own(const aim_ctx* c) { return (c->precision == AIM_C64) == (sizeof(C) == sizeof(float2)); }
  static int zw(const aim_ctx* c) { return own(c) && c->plan.zw ? c->plan.zw : def_zw(c); }
  static int cw(const aim_ctx* c) { return own(c) && c->plan.cw ? c->plan.cw : def_cw(); }
  static int rp(const aim_ctx* c) { return own(c) && c->plan.rp ? c->plan.rp : def_rp(c); }
  static int ypb(const aim_ctx* c) { return own(c) && c->plan.ypb ? c->plan.ypb : def_ypb(c); }
  // candidates the autotuner times: z tiles of x-adjacent columns (w divides L), y tiles
  static std::vector<int> zwidths(const aim_ctx* c) {
    std::vector<int> v;
    for (int w : {8, 16, 32, 64})
      if (w <= L && L % w == 0 && smem_z(c->LZ, w) <= kPlanSmemMax) v.push_back(w);
    return v;
  }
  static std::vector<int> ywidths() {
    std::vector<int> v;
    for (int w : {8, 16, 32, 64})
      if (w <= L && L % w == 0 && smem_y(w) <= kPlanSmemMax) v.push_back(w);
    return v;
  }
  static std::vector<int> rps(const aim_ctx* c) {
    std::vector<int> v;
    if (kxm(c)) {
      for (int r : {1, 2, 4, 8, 16})
        if (r <= c->N) v.push_back(r);
    } else {
      for (int r : {2, 4, 8, 16, 32, 64})
        if (smem_x(r) <= 100 * 1024) v.push_back(r);
    }
    return v;
  }
  static std::vector<int> ypbs(const aim_ctx* c) {
    std::vector<int> v;
    for (int y : {1, 2, 4, 8})
      if (y <= c->N && smem_anterp(y, 1, kxm(c)) <= 100 * 1024) v.push_back(y);
    return v;
  }
  // rows per block of the x passes: the largest instantiated count not above the plan's
  template <class F>
  static void with_rows(int r, int most, F&& f) {
    r = std::min(r, most);
    if (r >= 16) f(std::integral_constant<int, 16>{});
    else if (r >= 8) f(std::integral_constant<int, 8>{});
    else if (r >= 4) f(std::integral_constant<int, 4>{});
    else if (r >= 2) f(std::integral_constant<int, 2>{});
    else f(std::integral_constant<int, 1>{});
  }

  // stage i + forward x and y passes: v[nb][ns] (optionally times dinv) -> slab [nb][4][nz][L][L]
  // dinv non-null asks for the context's right preconditioner: the diagonal dinv, or the
  // near-zone SAI when the context built one
  static void prep(aim_ctx* c, int nb, const double2* v, const double2* dinv, VecSel vs, const int* active,
                   bool want_fp64) {
    const long long n = (long long)nb * c->ns;
    KScope ks(c, AIM_K_PREP);
    if (dinv && c->d_sai)
      launch_pdl(c->stream, dim3((unsigned)((n * 16 + 255) / 256)), dim3(256), 0, k_prep_sai<C>, v,
                 std::is_same<C, float2>::value ? (const float2*)c->d_vf : (const float2*)nullptr,
                 sel_sai(c, (C*)nullptr), (const int*)c->d_srowptr, (const int*)c->d_scol, vs, active, c->ns, nb,
                 reinterpret_cast<C*>(c->d_xs), want_fp64 ? c->d_xd : (double2*)nullptr);
    else
      launch_pdl(c->stream, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, k_prep<C>, v, dinv, vs, active, c->ns,
                 nb, reinterpret_cast<C*>(c->d_xs), want_fp64 ? c->d_xd : (double2*)nullptr);
  }

  // the active box (x, y, z node ranges): every pass touches only the grid lines that are
  // non-zero on input or needed on output; the buffers hold the box's nz z-planes only
  static int nbox(const aim_ctx* c, int d) { return c->box_hi[d] - c->box_lo[d] + 1; }
  static ZGeom zgeom(const aim_ctx* c) { return ZGeom{L, c->N, c->NZ}; }

  // anterpolation gather + forward x pass: d_xs -> A (rows of the active box)
  template <bool KXM>
  static void anterp_as(aim_ctx* c, int nb, const int* active) {
    const int most = std::min(8, L / 2), nyb = nbox(c, 1);
    // a complex64 batch in pairs (two right-hand sides per block share the coefficient loads)
    // where the pairs fill the chip four times with 4 rows per block; else 4 lanes per node
    // (3 waves, 1160 unknowns: 8.6 us against 12.7 in pairs; 64 waves, 7680 unknowns: 533 us against
    // 469 in pairs with one partial sum per node, about 520 with the four that keep the order).  complex128 keeps the 4 lanes: the pairs' partial sums take too many registers
    constexpr bool kPairs = std::is_same<C, float2>::value;
    const long long pairs = (long long)((nb + 1) / 2) * c->NZ * ((nyb + 3) / 4);
    const int bb = kPairs && nb > 1 && pairs >= 4 * 152 ? 2 : 1;
    int yp = ypb(c);
    while (yp > 1 && smem_anterp(yp, bb, KXM) > (size_t)kPlaneSmemMax) yp /= 2;
    with_rows(yp, most, [&](auto yt) {
      constexpr int YB = decltype(yt)::value;
      if constexpr (YB <= 8 && YB <= L / 2) {
        auto go = [&](auto bt) {
          constexpr int BB = decltype(bt)::value;
          auto kern = k_anterp<L, YB, BB, KXM, C>;
          const size_t sm = smem_anterp(YB, BB, KXM);
          if (sm > (size_t)kPlaneSmemMax) throw AimError{AIM_ERR_ARG, "launch plan: anterpolation tile"};
          smem_opt_in(kern, sm);
          launch_pdl(c->stream, dim3((nb + BB - 1) / BB, ((KXM ? c->N : nyb) + YB - 1) / YB, c->NZ), dim3(256), sm,
                     kern, (const int*)c->d_arow, (const int*)c->d_anode, (const int*)c->d_aptr,
                     (const int*)c->d_nidx, ncoef(c), reinterpret_cast<const C*>(c->d_xs), active, nb,
                     reinterpret_cast<C*>(c->d_A), twiddles(c), c->box_lo[1], nyb, c->NZ);
        };
        if constexpr (kPairs) {
          if (bb == 2) return go(std::integral_constant<int, 2>{});
        }
        go(std::integral_constant<int, 1>{});
      }
    });
  }
  static void anterp_x(aim_ctx* c, int nb, const int* active) {
    KScope ks(c, AIM_K_ANTERP_XFFT);
    if constexpr (L <= 256) {
      if (kxm(c)) return anterp_as<true>(c, nb, active);
    }
    anterp_as<false>(c, nb, active);
  }

  template <bool INV>
  static void ypipe(aim_ctx* c, int nb, const float2* in, float2* out) {
    using Y = YPipe<L, INV>;
    const int ntiles = nb * 4 * c->NZ * (L / Y::W), lo = c->box_lo[1], hi = c->box_hi[1];
    const long long half = (long long)c->N * L, full = (long long)L * L;
    auto kern = k_ypipe<L, INV>;
    smem_opt_in(kern, Y::smem);
    launch_pdl(c->stream, dim3(std::min(ntiles, 152 * Y::blocks)), dim3(Y::NT), Y::smem, kern, in, out, ntiles,
               INV ? 0 : lo, INV ? L - 1 : hi, lo, hi, INV ? full : half, INV ? half : full, twiddles(c));
  }

  // forward y pass (pruned input): A -> slab
  static void y_fwd(aim_ctx* c, int nb, C* slab) {
    static_assert(two_step_len(L), "every supported padded length has a two-step plan");
    const int N = c->N, nz = c->NZ;
    const C* A = reinterpret_cast<const C*>(c->d_A);
    KScope ks(c, AIM_K_YFFT_FWD);
    if constexpr (ypipe_len<L, C>()) return ypipe<false>(c, nb, A, slab);
    with_width(cw(c), [&](auto wt) {
      constexpr int CW = decltype(wt)::value;
      if constexpr (CW <= L) {
        const size_t sm = smem_y(CW);
        smem_opt_in(k_cols_p2<L, CW, false, C, true>, sm);
        // lines (plane, x): inputs y in the box, all L outputs
        launch_pdl(c->stream, dim3(L / CW, nz, nb * 4), dim3(256), sm, k_cols_p2<L, CW, false, C, true>, A, slab,
                   c->box_hi[1] + 1, L, (long long)L, (long long)L, L, (long long)N * L, (long long)L * L,
                   (long long)nz * N * L, (long long)nz * L * L, twiddles(c), c->box_lo[1], 0, 0);
      } else {
        throw AimError{AIM_ERR_ARG, "launch plan: tile wider than the line"};
      }
    });
  }

  // inverse y pass (pruned output): Bf -> A
  static void y_inv(aim_ctx* c, int nb) {
    const int N = c->N, nz = c->NZ;
    KScope ks(c, AIM_K_YFFT_INV);
    if constexpr (ypipe_len<L, C>())
      return ypipe<true>(c, nb, reinterpret_cast<const C*>(c->d_Bf), reinterpret_cast<C*>(c->d_A));
    with_width(cw(c), [&](auto wt) {
      constexpr int CW = decltype(wt)::value;
      if constexpr (CW <= L) {
        const size_t sm = smem_y(CW);
        smem_opt_in(k_cols_p2<L, CW, true, C>, sm);
        // lines (plane, x): all L inputs, outputs y in the box
        launch_pdl(c->stream, dim3(L / CW, nz, nb * 4), dim3(256), sm, k_cols_p2<L, CW, true, C>,
                   (const C*)c->d_Bf, reinterpret_cast<C*>(c->d_A), L, c->box_hi[1] + 1, (long long)L, (long long)L, L,
                   (long long)L * L, (long long)N * L, (long long)nz * L * L, (long long)nz * N * L, twiddles(c), 0,
                   c->box_lo[1], 0);
      } else {
        throw AimError{AIM_ERR_ARG, "launch plan: tile wider than the line"};
      }
    });
  }

  // inverse x pass (pruned output): A -> P, the rows of the active box, outputs x in the box
  static void x_inv(aim_ctx* c, int nb) {
    if constexpr (L <= 256) {
      if (kxm(c)) {
        KScope ks(c, AIM_K_XFFT_INV);
        with_rows(rp(c), std::min(16, L / 2), [&](auto yt) {
          constexpr int YB = decltype(yt)::value;
          if constexpr (YB <= L / 2) {
            const size_t sm = smem_xinv(YB);
            smem_opt_in(k_xinv<L, YB, C>, sm);
            launch_pdl(c->stream, dim3((nbox(c, 1) + YB - 1) / YB, c->NZ, nb * 4), dim3(256), sm, k_xinv<L, YB, C>,
                       (const C*)c->d_A, reinterpret_cast<C*>(c->d_P), twiddles(c), c->box_lo[1], nbox(c, 1), c->NZ);
          }
        });
        return;
      }
    }
    const int N = c->N, r = rp(c), nz = c->NZ, ny = nbox(c, 1), nrows = nb * 4 * nz * ny;
    const size_t sm = smem_x(r);
    smem_opt_in(k_rows_p2<L, true, C>, sm);
    KScope ks(c, AIM_K_XFFT_INV);
    launch_pdl(c->stream, dim3((nrows + r - 1) / r), dim3(256), sm, k_rows_p2<L, true, C>, (const C*)c->d_A,
               reinterpret_cast<C*>(c->d_P), nrows, L, c->box_hi[0] + 1, (long long)L, (long long)N, twiddles(c), r,
               RowBox{nz, ny, 0, c->box_lo[1], nz, N}, c->box_lo[0]);
  }

  static void forward_slab(aim_ctx* c, int nb, const double2* v, const double2* dinv, const int* active, C* slab,
                           VecSel vs = VecSel(), bool want_fp64 = false) {
    prep(c, nb, v, dinv, vs, active, want_fp64);
    anterp_x(c, nb, active);
    if (!kxm(c)) y_fwd(c, nb, slab);
  }

  // the spectra of `slots` vectors v[slots][nb][ns] in one launch of each pass (kx-major
  // grids; their grid stages use the batch buffers d_Ab, d_xsb)
  static void forward_slots(aim_ctx* c, int slots, int nb, const double2* v, C* dst, size_t slot_elems) {
    struct Swap {  // the batch buffers stand in for the context's for the duration
      aim_ctx* c;
      void *A, *xs;
      explicit Swap(aim_ctx* c_) : c(c_), A(c_->d_A), xs(c_->d_xs) {
        c->d_A = c->d_Ab;
        c->d_xs = c->d_xsb;
      }
      ~Swap() {
        c->d_A = A;
        c->d_xs = xs;
      }
    } sw(c);
    prep(c, slots * nb, v, nullptr, VecSel(), nullptr, false);
    anterp_x(c, slots * nb, nullptr);
    KScope ks(c, AIM_K_ZFWD);
    plane_launch<C>(c, nb, PLANE_FWD, 0, nullptr, dst, slots, slot_elems);
  }

  // inverse y and x passes: Bf slab -> P, then interpolation + near terms
  static void backward(aim_ctx* c, int nb, const NearList& nl, const double2* base, double sign, const int* active,
                       double2* y, VecSel ys = VecSel()) {
    if (!kxm(c)) y_inv(c, nb);
    x_inv(c, nb);
    interp(c, nb, reinterpret_cast<const C*>(c->d_P), nl, base, sign, active, y, ys);
  }

  static void interp(aim_ctx* c, int nb, const C* P, const NearList& nl, const double2* base, double sign,
                     const int* active, double2* y, VecSel ys = VecSel()) {
    KScope ks(c, AIM_K_INTERP_NEAR);
    const int br = 8 * interp_rows(c->ns);
    const unsigned nrb = (unsigned)((c->ns + br - 1) / br);
    if (nrb > 65535u) throw AimError{AIM_ERR_ARG, "interpolation: more than 2 097 120 RWGs"};
    launch_pdl(c->stream, dim3((unsigned)nb, nrb), dim3(256), 0,
               interp_rows(c->ns) == 4 ? k_interp_near<C, 4> : k_interp_near<C, 1>, P, (const int*)c->d_anchor,
               (const int*)c->d_order, lam(c), c->N, c->NZ, c->box_lo[2], c->ns, nb, (const int*)c->d_rowptr,
               (const int*)c->d_col, nl, base, sign, active, y, ys, c->dotfuse);
  }

  // size of one kernel-spectrum octant [LZ/2 + 1][N + 1][N + 1]
  static size_t octant(const aim_ctx* c) { return (size_t)(c->N + 1) * (c->N + 1) * (c->LZ / 2 + 1); }

  static void zconv(aim_ctx* c, int nb, int m, const int* active) {
    KScope ks(c, AIM_K_ZCONV);
    if (kxm(c)) return plane_launch<C>(c, nb, PLANE_CONV, m, active, nullptr, 1, 0);
    C* Bf = reinterpret_cast<C*>(c->d_Bf);
    const C* G = kspec(c) + (size_t)m * 2 * octant(c);
    with_zlen(c->LZ, [&](auto lz) {
      constexpr int LZ = decltype(lz)::value;
      if constexpr (zwarp_len<L, LZ, C>()) {
        constexpr size_t sm = ZWarp<LZ>::smem;
        smem_opt_in(k_zwarp<LZ, Z_CONV>, sm);
        launch_pdl(c->stream, dim3(L / (ZWarp<LZ>::CW * ZWarp<LZ>::NW), L), dim3(32 * ZWarp<LZ>::NW), sm,
                   k_zwarp<LZ, Z_CONV>, Bf, G, zgeom(c), nb, active,
                   ztwiddles(c), SlabList{});
      } else if constexpr (LZ <= L && !plane_always<L, LZ, C>()) {
        with_width(zw(c), [&](auto wt) {
          constexpr int ZW = decltype(wt)::value;
          if constexpr (ZW <= L) {
            const size_t sm = smem_z(LZ, ZW);
            smem_opt_in(k_zconv_p2<LZ, ZW, C>, sm);
            launch_pdl(c->stream, dim3(nb * 4, L / ZW, L), dim3(kZThreads), sm, k_zconv_p2<LZ, ZW, C>, Bf, G,
                       zgeom(c), active, ztwiddles(c));
          } else {
            throw AimError{AIM_ERR_ARG, "launch plan: tile wider than the line"};
          }
        });
      } else {
        throw AimError{AIM_ERR_ARG, "z transform longer than the padded length"};
      }
    });
    AIM_CHECK_LAUNCH();
  }

  // Autotuner: time every candidate launch shape of each pass on this context's buffers
  // (nb = batch_max right-hand sides, the contents are irrelevant to the timing) and keep
  // the fastest.  Each pass's arithmetic per line is the same for every shape.
  static void tune(aim_ctx* c) {
    const int nb = c->batch_max;
    cudaEvent_t e0, e1;
    AIM_CUDA(cudaEventCreate(&e0));
    AIM_CUDA(cudaEventCreate(&e1));
    auto time_ms = [&](const std::function<void()>& launch) {
      launch();  // first launch: shared-memory attribute and warm-up
      float best = 1e30f;
      for (int r = 0; r < 3; ++r) {
        AIM_CUDA(cudaEventRecord(e0, c->stream));
        launch();
        AIM_CUDA(cudaEventRecord(e1, c->stream));
        AIM_CUDA(cudaEventSynchronize(e1));
        float ms = 0;
        AIM_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        best = std::min(best, ms);
      }
      return best;
    };
    KPlan& p = c->plan;
    auto pick = [&](int& field, const std::vector<int>& cand, const std::function<void()>& launch) {
      float best = 1e30f;
      int arg = cand.empty() ? 0 : cand[0];
      for (int v : cand) {
        field = v;
        const float t = time_ms(launch);
        if (t < best) {
          best = t;
          arg = v;
        }
      }
      field = arg;
    };
    // k_plane, k_zwarp and k_ypipe have one shape: the fields keep the defaults there
    bool zwarp = false;
    with_zlen(c->LZ, [&](auto lz) { zwarp = zwarp_len<L, decltype(lz)::value, C>(); });
    if (kxm(c) || zwarp)
      p.zw = def_zw(c);
    else
      pick(p.zw, zwidths(c), [&] { zconv(c, nb, 0, nullptr); });
    if (kxm(c) || ypipe_len<L, C>())
      p.cw = def_cw();
    else
      pick(p.cw, ywidths(), [&] {
        y_fwd(c, nb, reinterpret_cast<C*>(c->d_Bf));
        y_inv(c, nb);
      });
    pick(p.rp, rps(c), [&] { x_inv(c, nb); });
    pick(p.ypb, ypbs(c), [&] { anterp_x(c, nb, nullptr); });
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }

  // forward z-FFT of the slab in Bf into the z-spectral history layout at dst
  // (power-of-two z lengths only)
  static void zfwd(aim_ctx* c, int nb, C* dst) {
    if (kxm(c)) {
      KScope ks(c, AIM_K_ZFWD);
      return plane_launch<C>(c, nb, PLANE_FWD, 0, nullptr, dst, 1, 0);
    }
    with_zlen(c->LZ, [&](auto lz) {
      constexpr int LZ = decltype(lz)::value;
      if constexpr (pow2_len(LZ) && LZ <= L && !plane_always<L, LZ, C>()) {
        constexpr int ZW = zcol_width<LZ, C>();
        const size_t sm = smem_z(LZ, ZW);
        KScope ks(c, AIM_K_ZFWD);
        smem_opt_in(k_zfwd_spec<LZ, ZW, C>, sm);
        k_zfwd_spec<LZ, ZW, C><<<dim3(L / ZW, L, nb * 4), kZThreads, sm, c->stream>>>(
            reinterpret_cast<const C*>(c->d_Bf), dst, zgeom(c), ztwiddles(c));
        AIM_CHECK_LAUNCH();
      } else {
        throw AimError{AIM_ERR_ARG, "z-spectral history needs a power-of-two z length"};
      }
    });
  }

  static void zrhs(aim_ctx* c, int nb, const SlabList& sl, C* scratch) {
    C* Bf = reinterpret_cast<C*>(c->d_Bf);
    KScope ks(c, AIM_K_ZRHS);
    if (kxm(c)) return plane_rhs<C>(c, nb, sl, scratch);
    with_zlen(c->LZ, [&](auto lz) {
      constexpr int LZ = decltype(lz)::value;
      if constexpr (zwarp_len<L, LZ, C>()) {
        constexpr size_t sm = ZWarp<LZ>::smem;
        smem_opt_in(k_zwarp<LZ, Z_RHS>, sm);
        launch_pdl(c->stream, dim3(L / (ZWarp<LZ>::CW * ZWarp<LZ>::NW), L, nb * 4), dim3(32 * ZWarp<LZ>::NW),
                   sm, k_zwarp<LZ, Z_RHS>, Bf, kspec(c), zgeom(c), nb,
                   (const int*)nullptr, ztwiddles(c), sl);
      } else if constexpr (LZ <= L && !plane_always<L, LZ, C>()) {
        if constexpr (pow2_len(LZ) && LZ <= 256 && L <= 256 && std::is_same<C, float2>::value) {
          // the spectra's ring slots (the march and aim_rhs keep every history slab in the ring)
          const size_t slab = op_slab_bytes(c, c->batch_max);
          SlabRing sr{};
          sr.n = sl.n;
          bool in_ring = c->ring_tma && sl.n > 0;
          for (int i = 0; i < sl.n && in_ring; ++i) {
            const long long off = (const char*)sl.p[i] - (const char*)c->d_ring;
            in_ring = off >= 0 && off % (long long)slab == 0 && off / (long long)slab < c->n_delays;
            sr.slot[i] = in_ring ? (int)(off / (long long)slab) : 0;
            sr.m[i] = sl.m[i];
          }
          if (in_ring) {
            constexpr int ZW = L < 16 ? L : 16;
            const size_t sm = 128 + (2 * LZ * ZW + LZ + LZ * ZW) * sizeof(C);
            smem_opt_in(k_zrhs_spec_tma<LZ, ZW>, sm);
            k_zrhs_spec_tma<LZ, ZW><<<dim3(L / ZW, L, nb * 4), kZThreads, sm, c->stream>>>(
                c->ring_map, sr, kspec(c), zgeom(c), Bf, ztwiddles(c), c->d_err);
            AIM_CHECK_LAUNCH();
            return;
          }
        }
        if constexpr (pow2_len(LZ)) {
          // 16 columns per tile: one step-B item per thread, so the delay sum held in
          // registers stays at one radix-R2 slice
          constexpr int ZW = L < 16 ? L : 16;
          const size_t sm = smem_z(LZ, ZW);
          smem_opt_in(k_zrhs_spec<LZ, ZW, C>, sm);
          k_zrhs_spec<LZ, ZW, C><<<dim3(L / ZW, L, nb * 4), kZThreads, sm, c->stream>>>(sl, kspec(c), zgeom(c), Bf,
                                                                                      ztwiddles(c));
        } else {
          // one step-B item per thread, the delay sum held in registers
          constexpr int ZW = zsplit_r1<LZ>() <= 16 ? 16 : 8;
          const size_t sm = smem_z(LZ, ZW);
          smem_opt_in(k_zrhs_2s<LZ, ZW, C>, sm);
          k_zrhs_2s<LZ, ZW, C><<<dim3(nb * 4, L / ZW, L), kZThreads, sm, c->stream>>>(sl, kspec(c), zgeom(c), Bf,
                                                                                    ztwiddles(c));
        }
        AIM_CHECK_LAUNCH();
      } else {
        throw AimError{AIM_ERR_ARG, "z transform longer than the padded length"};
      }
    });
  }

  // blocked right-hand side: pending z-spectra -> slab of potentials in Bf (cleared)
  static void zinv_pending(aim_ctx* c, int nb, C* S) {
    if (kxm(c)) {
      // (cleared by a memset: with zeros stored between its loads the plane kernel took 204 us for
      // one vector on the 64^3 grid, the inverse and the memset take 39)
      KScope ks(c, AIM_K_ZINV_PENDING);
      plane_launch<C>(c, nb, PLANE_INV, 0, nullptr, S, 1, 0);
      AIM_CUDA(cudaMemsetAsync(S, 0, op_slab_bytes(c, nb), c->stream));
      return;
    }
    with_zlen(c->LZ, [&](auto lz) {
      constexpr int LZ = decltype(lz)::value;
      if constexpr (pow2_len(LZ) && LZ <= L && !plane_always<L, LZ, C>()) {
        constexpr int ZW = L < 16 ? L : 16;
        const size_t sm = smem_z(LZ, ZW);
        KScope ks(c, AIM_K_ZINV_PENDING);
        smem_opt_in(k_zinv_pending<LZ, ZW, C>, sm);
        k_zinv_pending<LZ, ZW, C><<<dim3(L / ZW, L, nb * 4), kZThreads, sm, c->stream>>>(
            S, zgeom(c), reinterpret_cast<C*>(c->d_Bf), ztwiddles(c));
        AIM_CHECK_LAUNCH();
      } else {
        throw AimError{AIM_ERR_ARG, "the blocked right-hand side needs a power-of-two z length"};
      }
    });
  }

  static void block_square(aim_ctx* c, int nb, const BlockSquare& sq) {
    const long long n = (long long)nb * 4 * c->LZ * L * L;
    const int grid = (int)std::min<long long>((n + 255) / 256, 152LL * 8);
    const int per = (grid + nb * 4 - 1) / (nb * 4);  // blocks per right-hand side and component
    KScope ks(c, AIM_K_BLOCK_SQUARE);
    auto go = [&](auto bt) {
      constexpr int B = decltype(bt)::value;
      if (kxm(c))
        with_zlen(c->LZ, [&](auto lz) {
          if constexpr (plane_fits<L, decltype(lz)::value, C>())
            k_block_square_plane<B, C><<<dim3(per, nb * 4), 256, 0, c->stream>>>(
                sq, plane_spec(c), plane_order<L, decltype(lz)::value, C>(), c->n_delays);
        });
      else
        k_block_square<B, C><<<grid, 256, 0, c->stream>>>(sq, kspec(c), zgeom(c), c->LZ, c->n_delays, n);
    };
    switch (sq.b) {
      case 1: go(std::integral_constant<int, 1>{}); break;
      case 2: go(std::integral_constant<int, 2>{}); break;
      case 4: go(std::integral_constant<int, 4>{}); break;
      case 8: go(std::integral_constant<int, 8>{}); break;
      case 16: go(std::integral_constant<int, 16>{}); break;
      default: throw AimError{AIM_ERR_ARG, "blocked right-hand side: square size"};
    }
    AIM_CHECK_LAUNCH();
  }

  static const C* twiddles(aim_ctx* c) { return sel_tw(c, (C*)nullptr); }
  static const C* ztwiddles(aim_ctx* c) { return sel_twz(c, (C*)nullptr); }
  static const C* kspec(aim_ctx* c) { return sel_kspec(c, (C*)nullptr); }
  static const C* plane_spec(aim_ctx* c) { return sel_plane(c, (C*)nullptr); }
  static const typename Real<C>::F4* ncoef(aim_ctx* c) { return sel_ncoef(c, (C*)nullptr); }
  static const typename Real<C>::T* lam(aim_ctx* c) { return sel_lam(c, (C*)nullptr); }
};
