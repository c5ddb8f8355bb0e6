// The y and z passes of the operator fused over one kx plane.
//
// After the forward x-FFT the grid of one (right-hand side, component) is a stack of L
// planes, one per kx, and nothing couples them until the inverse x-FFT.  k_plane holds one
// plane in shared memory and runs on it the forward y-FFT, the forward z-FFT, the product
// with the kernel spectrum, the inverse z-FFT and the inverse y-FFT, so the doubly padded
// slab never reaches memory: the plane is read and written once in its unpadded size
// [nz][N].  The x passes therefore store the grid kx-major,
//   A [b][c][kx < L][z < nz][y < N],
// and a plane is one contiguous run.
//
// Each length is split R1 x R2 (n = R2 n1 + n2, k = k1 + R1 k2).  A warp owns whole lines
// (rows z of the y-FFT, columns ky of the z-FFT), so the exchange between the two radix
// steps needs only __syncwarp; the block synchronises twice per plane, where the lines
// change direction.  The spectrum of a row stays in the order the second step leaves it
// in (position p = k1 R2 + k2 holds ky = k1 + R1 k2): the inverse y-FFT starts from the
// same order and the kernel spectrum is tabulated in it, so nothing is ever reordered.
// The z spectrum exists in registers only: lane u = k1 CW + col of a group of CW columns
// holds the R2 values kz = k1 + R1 k2 of its column, and the kernel spectrum and the
// history spectra are stored in exactly that order,
//   [group][k2 / 2][u][k2 & 1],
// one coalesced 16-byte load per lane for every two values.
//
// What bounds it: shared-memory bandwidth in complex64 (about 10 700 wavefronts per 128 x 128
// plane, 83 % of the cycles of the L1 pipe in use), FP64 arithmetic in complex128.  64 waves
// on the 64^3 grid, complex64: y, z and inverse y passes 2380 us as three kernels, which
// together moved 10.4 GB, 1580 us here, moving 2.1 GB.  A z step held in registers (two
// lanes or two warps per column, 64 values each) crosses shared memory half as often but
// leaves too few warps: when the exchange form took 1620 us it took 1580 to 1740, and 93 against
// 86 us for the product of a single wave (85 us now), so it is not used.  The next kernel of the
// chain is not released early (griddepcontrol.launch_dependents at the start): blocks waiting
// beside a running kernel made a chain of small kernels slower, 108 us against the 62 us that a
// product at 480 unknowns took then (48 us now).
#pragma once
#include "fft.cuh"
#include "fft_kernels.cuh"

constexpr int kPlaneSmemMax = 227 * 1024;  // shared memory a block can opt in to

// radix split of a length (R1 for the step next to the padding, whose zero half is pruned)
__host__ __device__ constexpr int pl_r1(int L) {
  return L == 16 ? 4 : L == 32 ? 8 : L == 64 ? 8 : L == 144 ? 12 : (L == 128 || L == 192 || L == 256) ? 16 : 0;
}
__host__ __device__ constexpr int pl_r2(int L) { return pl_r1(L) ? L / pl_r1(L) : 0; }
// the first pitch >= p that is r mod 16
__host__ __device__ constexpr int pl_round(int p, int r) {
  while (p % 16 != r) ++p;
  return p;
}

// Shapes of the plane kernel for one size.
template <int L, int LZ, class C>
struct PlaneCfg {
  static constexpr bool ok = pl_r1(L) > 0 && pl_r1(LZ) > 0 && LZ <= L;
  static constexpr int Y1 = pl_r1(L), Y2 = pl_r2(L), Z1 = pl_r1(LZ), Z2 = pl_r2(LZ);
  static constexpr int NW = L <= 32 ? 4 : (L == 192 && LZ == 192) ? 16 : 8;  // warps
  static constexpr int RW = Y2 == 4 ? 8 : Y2 == 16 ? 2 : 4;  // rows a warp takes at a time
  // columns a warp takes at a time
  static constexpr int CW = Z2 == 4 ? 8 : (Z2 == 16 || LZ == 192) ? 2 : 4;
  // Row pitch of the slab.  A row is Y1 blocks of Y2 values; the second y step reads one
  // block per lane, so a block is padded by one element.  Rows are 4 (2 where a warp takes
  // 2 columns) mod 16 apart, so the rows of a column group fall in different bank groups.
  static constexpr int YB = Y2 + 1;
  static constexpr int PY = ok ? pl_round(Y1 * YB, CW == 2 ? 2 : 4) : 0;
  static constexpr int PZ = ok ? pl_round(Z1 * (Z2 + 1), 4) : 0;  // exchange buffer pitch
  static constexpr int TY = Y1 * (Y2 + 1), TZ = Z1 * (Z2 + 1);    // twiddle tables
  static constexpr int SCR = CW * PZ;                             // exchange elements per warp
  static constexpr size_t smem = ok ? ((size_t)(L == LZ ? TY : TY + TZ) + (size_t)(LZ / 2) * PY + (size_t)NW * SCR) * sizeof(C) : 0;
  // blocks per SM the register allocation aims at (shared memory allows as many)
  static constexpr int by_smem = ok ? (int)((size_t)(228 * 1024) / (smem + 1024)) : 1;
  // A plane of complex128 has to leave room for a second one on its SM: alone, its load, FP64
  // and store phases follow one another, and the separate passes are as fast or faster (one
  // vector, us per product, plane against separate: 64^3 with 128 points in z 1319 and 1186,
  // with 64 points 583 and 518, 96^3 with 64 points 1537 and 1293; four vectors 4557 and 4503,
  // 1919 and 1856, 5220 and 4887; 16 vectors on 64^3 17.5 and 17.7 ms).
  static constexpr bool fits = ok && smem <= (size_t)kPlaneSmemMax && (sizeof(C) == 8 || by_smem >= 2);
  static constexpr int threads = (Y1 == 16 || Z1 == 16) ? (sizeof(C) == 8 ? 512 : 256) : (sizeof(C) == 8 ? 1024 : 512);
  static constexpr int most = threads / (32 * NW) < 1 ? 1 : threads / (32 * NW);
  static constexpr int blocks = by_smem < 1 ? 1 : by_smem < most ? by_smem : most;
};
template <int L, int LZ, class C>
constexpr bool plane_fits() { return PlaneCfg<L, LZ, C>::fits; }

// Order of the spectra, for set-up and the elementwise kernels.  Column position p = k1 Y2 + k2
// of a row holds ky = k1 + Y1 k2; unit u = k1z cw + col of a group, values kz = k1z + Z1 k2.
// The spectrum is even in ky: where a group lies inside one k1 block, the groups of k1 > Y1/2
// are those of Y1 - k1 with the columns reversed, and only `stored` groups are tabulated.
struct PlaneOrder {
  int L, LZ, y1, y2, z1;
  int cw, h, n, stored;  // columns per group, groups per k1 block (0: not folded), groups, tabulated groups
};
template <int L, int LZ, class C>
__host__ __device__ constexpr PlaneOrder plane_order() {
  using P = PlaneCfg<L, LZ, C>;
  PlaneOrder o{};
  o.L = L, o.LZ = LZ, o.y1 = P::Y1, o.y2 = P::Y2, o.z1 = P::Z1;
  o.cw = P::CW;
  o.n = L / P::CW;
  o.h = P::Y2 % P::CW == 0 ? P::Y2 / P::CW : 0;
  o.stored = o.h ? (P::Y1 / 2 + 1) * o.h : o.n;
  return o;
}
// tabulated elements of one kx, and of one delay: [kind 2][kx <= L/2][...]
__host__ __device__ constexpr size_t plane_g_elems(const PlaneOrder& o) { return (size_t)o.stored * o.cw * o.LZ; }
__host__ __device__ constexpr size_t plane_spec_elems(const PlaneOrder& o) {
  return (size_t)2 * (o.L / 2 + 1) * plane_g_elems(o);
}

// ---------------------------------------------------------------- two adjacent values at a time
__device__ __forceinline__ void ld2(const float2* p, float2& a, float2& b) {
  const float4 q = __ldg(reinterpret_cast<const float4*>(p));
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld2(const double2* p, double2& a, double2& b) {
  a = __ldg(p);
  b = __ldg(p + 1);
}
// (through L2 only: history spectra are read once)
__device__ __forceinline__ void ld2_stream(const float2* p, float2& a, float2& b) {
  const float4 q = __ldcs(reinterpret_cast<const float4*>(p));
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld2_stream(const double2* p, double2& a, double2& b) {
  a = __ldcs(p);
  b = __ldcs(p + 1);
}
__device__ __forceinline__ void st2(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st2(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// ---------------------------------------------------------------- the plane kernel
enum { PLANE_CONV = 0,  // A <- inverse(G_m . forward(A))
       PLANE_FWD = 1,   // S <- forward(A)
       PLANE_INV = 2    // A <- inverse(S)
};

template <int L, int LZ, class C>
struct PlaneFFT : PlaneCfg<L, LZ, C> {
  using Cfg = PlaneCfg<L, LZ, C>;
  using Cfg::CW;
  using Cfg::NW;
  using Cfg::PY;
  using Cfg::PZ;
  using Cfg::RW;
  using Cfg::Y1;
  using Cfg::Y2;
  using Cfg::YB;
  using Cfg::Z1;
  using Cfg::Z2;
  static constexpr int UA = CW * Z2, UB = CW * Z1;          // units of the two z steps per group
  static constexpr int QA = (UA + 31) / 32, QB = (UB + 31) / 32;
  static constexpr int N = L / 2;

  // rows z0 .. z0 + RW - 1 < nz of the plane: forward y-FFT into the slab
  static __device__ __forceinline__ void y_forward(const C* __restrict__ A, C* slab, const C* tw, int z0, int nz) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < (RW * Y2 + 31) / 32; ++q) {
      const int u = lane + 32 * q, n2 = u % Y2;
      int r = u / Y2;
      if (RW == 4) r = ((r & 1) << 1) | (r >> 1);  // the two rows of a half-warp 8 slots apart
      if (((RW * Y2) % 32 == 0 || u < RW * Y2) && z0 + r < nz) {
        const C* src = A + (size_t)(z0 + r) * N + n2;
        C v[Y1];
#pragma unroll
        for (int n1 = 0; n1 < Y1 / 2; ++n1) v[n1] = src[Y2 * n1];
        HalfDFT<Y1, false, C>::in(v);
        C* dst = slab + (z0 + r) * PY + n2;
#pragma unroll
        for (int k1 = 0; k1 < Y1; ++k1) dst[k1 * YB] = k1 ? v[k1] * tw[k1 * (Y2 + 1) + n2] : v[k1];
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < (RW * Y1 + 31) / 32; ++q) {
      const int u = lane + 32 * q, k1 = u % Y1, r = u / Y1;
      if (((RW * Y1) % 32 == 0 || u < RW * Y1) && z0 + r < nz) {
        C* t = slab + (z0 + r) * PY + k1 * YB;
        C v[Y2];
#pragma unroll
        for (int n2 = 0; n2 < Y2; ++n2) v[n2] = t[n2];
        DFTL<Y2, L, false, C>::run(v, tw);
#pragma unroll
        for (int k2 = 0; k2 < Y2; ++k2) t[k2] = v[k2];
      }
    }
  }

  // the inverse: rows of the slab to the plane
  static __device__ __forceinline__ void y_inverse(C* __restrict__ A, C* slab, const C* tw, int z0, int nz) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < (RW * Y1 + 31) / 32; ++q) {
      const int u = lane + 32 * q, k1 = u % Y1, r = u / Y1;
      if (((RW * Y1) % 32 == 0 || u < RW * Y1) && z0 + r < nz) {
        C* t = slab + (z0 + r) * PY + k1 * YB;
        C v[Y2];
#pragma unroll
        for (int k2 = 0; k2 < Y2; ++k2) v[k2] = t[k2];
        DFTL<Y2, L, true, C>::run(v, tw);
#pragma unroll
        for (int n2 = 0; n2 < Y2; ++n2) t[n2] = n2 ? v[n2] * conjc(tw[k1 * (Y2 + 1) + n2]) : v[n2];
      }
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < (RW * Y2 + 31) / 32; ++q) {
      const int u = lane + 32 * q, n2 = u % Y2;
      int r = u / Y2;
      if (RW == 4) r = ((r & 1) << 1) | (r >> 1);
      if (((RW * Y2) % 32 == 0 || u < RW * Y2) && z0 + r < nz) {
        const C* t = slab + (z0 + r) * PY + n2;
        C v[Y1];
#pragma unroll
        for (int k1 = 0; k1 < Y1; ++k1) v[k1] = t[k1 * YB];
        HalfDFT<Y1, true, C>::out(v);
        C* dst = A + (size_t)(z0 + r) * N + n2;
#pragma unroll
        for (int n1 = 0; n1 < Y1 / 2; ++n1) dst[Y2 * n1] = v[n1];
      }
    }
  }

  // slab offset of column position p
  static __device__ __forceinline__ int pos(int p) { return (p / Y2) * YB + p % Y2; }

  // z step next to the padding, columns of group g, slab -> scr
  static __device__ __forceinline__ void z_step_a(const C* slab, C* scr, const C* tw, int g) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int u = lane + 32 * q, col = u % CW, n2 = u / CW;
      if (UA % 32 == 0 || u < UA) {
        const C* src = slab + n2 * PY + pos(g * CW + col);
        C v[Z1];
#pragma unroll
        for (int n1 = 0; n1 < Z1 / 2; ++n1) v[n1] = src[n1 * Z2 * PY];
        dft_half_in<Z1, LZ, false, C>(v, tw);
        C* dst = scr + col * PZ + n2;
#pragma unroll
        for (int k1 = 0; k1 < Z1; ++k1) dst[k1 * (Z2 + 1)] = k1 ? v[k1] * tw[k1 * (Z2 + 1) + n2] : v[k1];
      }
    }
  }
  static __device__ __forceinline__ void z_step_c(C* slab, const C* scr, int g) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int u = lane + 32 * q, col = u % CW, n2 = u / CW;
      if (UA % 32 == 0 || u < UA) {
        const C* src = scr + col * PZ + n2;
        C v[Z1];
#pragma unroll
        for (int k1 = 0; k1 < Z1; ++k1) v[k1] = src[k1 * (Z2 + 1)];
        dft_half_out<Z1, LZ, true, C>(v, nullptr);
        C* dst = slab + n2 * PY + pos(g * CW + col);
#pragma unroll
        for (int n1 = 0; n1 < Z1 / 2; ++n1) dst[n1 * Z2 * PY] = v[n1];
      }
    }
  }
  static __device__ __forceinline__ void b_forward(const C* t, const C* tw, C (&v)[Z2]) {
#pragma unroll
    for (int n2 = 0; n2 < Z2; ++n2) v[n2] = t[n2];
    DFTL<Z2, LZ, false, C>::run(v, tw);
  }
  static __device__ __forceinline__ void b_inverse(C* t, const C* tw, int k1, C (&v)[Z2]) {
    DFTL<Z2, LZ, true, C>::run(v, tw);
#pragma unroll
    for (int n2 = 0; n2 < Z2; ++n2) t[n2] = n2 ? v[n2] * conjc(tw[k1 * (Z2 + 1) + n2]) : v[n2];
  }

  // group g of the tabulated kernel spectrum and the unit index of u in it
  static __device__ __forceinline__ const C* g_group(const C* G, int g, bool& rev) {
    constexpr PlaneOrder o = plane_order<L, LZ, C>();
    rev = false;
    if constexpr (o.h > 0) {
      const int k1 = g / o.h;
      if (k1 > Y1 / 2) {
        rev = true;
        g = (Y1 - k1) * o.h + o.h - 1 - g % o.h;
      }
    }
    return G + (size_t)g * (CW * LZ);
  }
  static __device__ __forceinline__ int g_unit(int u, bool rev) {
    return rev ? u + CW - 1 - 2 * (u % CW) : u;
  }
};

template <class C>
struct PlaneArgs {
  C* A;              // [nb * 4][L][nz][N]
  C* S;              // FWD: spectra out; INV: spectra in
  const C* G;        // CONV: the tabulated spectrum of the delay
  int sbc;           // (right-hand side, component) pairs per spectrum; further ones go on
  size_t sstride;    // sstride elements after it (several delays in one launch)
  const int* active;
  const C* twy;
  const C* twz;
  int nz;
};

// Grid (nb * 4, L): the right-hand sides and components of one kx run together and share
// its kernel spectrum through L2; kx in mirror pairs (0, N, 1, L - 1, ...), whose spectra
// are the same.
template <int L, int LZ, class C, int MODE>
__global__ void __launch_bounds__(32 * PlaneCfg<L, LZ, C>::NW, (PlaneCfg<L, LZ, C>::blocks))
    k_plane(PlaneArgs<C> a) {
  using F = PlaneFFT<L, LZ, C>;
  constexpr PlaneOrder o = plane_order<L, LZ, C>();
  constexpr int NT = 32 * F::NW, N = L / 2;
  C* twz = reinterpret_cast<C*>(aim_smem);
  C* twy = L == LZ ? twz : twz + F::TZ;
  C* slab = twy + F::TY;
  C* scr = slab + (LZ / 2) * F::PY + (threadIdx.x >> 5) * F::SCR;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  load_twiddles2<F::Z1, F::Z2>(twz, a.twz);
  if (L != LZ) load_twiddles2<F::Y1, F::Y2>(twy, a.twy);
  if (MODE == PLANE_CONV || MODE == PLANE_FWD)  // the zero padding below the box
    for (int i = a.nz * F::PY + threadIdx.x; i < (LZ / 2) * F::PY; i += NT) slab[i] = C{};
  pdl_wait();
  const int bc = blockIdx.x, kx = zpass_row(blockIdx.y, N);
  if (a.active && !a.active[bc >> 2]) return;
  C* A = a.A + ((size_t)bc * L + kx) * a.nz * N;
  const int kind = (bc & 3) == 3 ? 1 : 0;
  const size_t goff = ((size_t)kind * (N + 1) + (kx <= N ? kx : L - kx)) * plane_g_elems(o);
  const size_t soff = (size_t)(bc / a.sbc) * a.sstride + ((size_t)(bc % a.sbc) * L + kx) * ((size_t)L * LZ);
  __syncthreads();
  if (MODE == PLANE_CONV || MODE == PLANE_FWD) {
    for (int z0 = warp * F::RW; z0 < a.nz; z0 += F::NW * F::RW) F::y_forward(A, slab, twy, z0, a.nz);
    __syncthreads();
  }
  for (int g = warp; g < L / F::CW; g += F::NW) {
    if constexpr (MODE == PLANE_CONV) {
      bool rev;
      const C* G = F::g_group(a.G + goff, g, rev);
      F::z_step_a(slab, scr, twz, g);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < F::QB; ++q) {
        const int u = lane + 32 * q, k1 = u / F::CW;
        if (F::UB % 32 == 0 || u < F::UB) {
          C* t = scr + (u % F::CW) * F::PZ + k1 * (F::Z2 + 1);
          const C* gp = G + 2 * F::g_unit(u, rev);
          C gk[F::Z2], v[F::Z2];
#pragma unroll
          for (int h = 0; h < F::Z2 / 2; ++h) ld2(gp + h * (2 * F::UB), gk[2 * h], gk[2 * h + 1]);
          F::b_forward(t, twz, v);
#pragma unroll
          for (int k2 = 0; k2 < F::Z2; ++k2) v[k2] = v[k2] * gk[k2];
          F::b_inverse(t, twz, k1, v);
        }
      }
      __syncwarp();
      F::z_step_c(slab, scr, g);
      __syncwarp();
    } else if constexpr (MODE == PLANE_FWD) {
      F::z_step_a(slab, scr, twz, g);
      __syncwarp();
      C* out = a.S + soff + (size_t)g * (F::CW * LZ);
#pragma unroll
      for (int q = 0; q < F::QB; ++q) {
        const int u = lane + 32 * q;
        if (F::UB % 32 == 0 || u < F::UB) {
          C v[F::Z2];
          F::b_forward(scr + (u % F::CW) * F::PZ + (u / F::CW) * (F::Z2 + 1), twz, v);
#pragma unroll
          for (int h = 0; h < F::Z2 / 2; ++h) st2(out + h * (2 * F::UB) + 2 * u, v[2 * h], v[2 * h + 1]);
        }
      }
      __syncwarp();
    } else {
      const C* in = a.S + soff + (size_t)g * (F::CW * LZ);
#pragma unroll
      for (int q = 0; q < F::QB; ++q) {
        const int u = lane + 32 * q, k1 = u / F::CW;
        if (F::UB % 32 == 0 || u < F::UB) {
          C v[F::Z2];
#pragma unroll
          for (int h = 0; h < F::Z2 / 2; ++h) {
            ld2_stream(in + h * (2 * F::UB) + 2 * u, v[2 * h], v[2 * h + 1]);
          }
          F::b_inverse(scr + (u % F::CW) * F::PZ + k1 * (F::Z2 + 1), twz, k1, v);
        }
      }
      __syncwarp();
      F::z_step_c(slab, scr, g);
      __syncwarp();
    }
  }
  if (MODE != PLANE_FWD) {
    __syncthreads();
    for (int z0 = warp * F::RW; z0 < a.nz; z0 += F::NW * F::RW) F::y_inverse(A, slab, twy, z0, a.nz);
  }
}

// Element i of the spectra of one (right-hand side, component), [kx][group]..., in the
// tabulated kernel spectrum of a kind.
// (at most 256^3 elements)
__device__ __forceinline__ size_t plane_g_index(const PlaneOrder& o, int i) {
  const int N = o.L / 2, per_kx = o.L * o.LZ, gsz = o.cw * o.LZ;
  const int kx = i / per_kx, q = i % per_kx;
  int g = q / gsz, r = q % gsz;
  const size_t base = (size_t)fold(kx, N) * plane_g_elems(o);
  if (o.h && g / o.h > o.y1 / 2) {  // the mirror group, columns reversed
    const int col = (r >> 1) % o.cw;
    r += 2 * (o.cw - 1 - 2 * col);
    g = (o.y1 - g / o.h) * o.h + o.h - 1 - g % o.h;
  }
  return base + (size_t)g * gsz + r;
}

// Delay sum of the right-hand side on z-spectra: out = sum_i G^_{m_i} . S_i, elementwise in
// the plane kernel's order (the spectra are read once and the sum goes through the plane
// kernel's inverse).  One thread takes two adjacent elements of one component; grid
// (pairs / 256, nb * 4).
template <class C>
__global__ void __launch_bounds__(256) k_spec_sum(const __grid_constant__ SlabList sl, const C* __restrict__ G,
                                                  PlaneOrder o, C* out) {
  const int per = o.L * o.L * o.LZ, i = 2 * (blockIdx.x * 256 + threadIdx.x);
  if (i >= per) return;
  const int bc = blockIdx.y;
  const C* gp = G + ((bc & 3) == 3 ? (size_t)(o.L / 2 + 1) * plane_g_elems(o) : 0);
  const size_t gm = plane_spec_elems(o), g0 = plane_g_index(o, i), g1 = plane_g_index(o, i + 1);
  const size_t q = (size_t)bc * per + i;
  C a0{}, a1{};
#pragma unroll 4
  for (int s = 0; s < sl.n; ++s) {
    C x0, x1;
    ld2_stream(reinterpret_cast<const C*>(sl.p[s]) + q, x0, x1);
    const C* g = gp + (size_t)sl.m[s] * gm;
    a0 += x0 * __ldg(g + g0);
    a1 += x1 * __ldg(g + g1);
  }
  st2(out + q, a0, a1);
}

// The tabulated kernel spectrum of one delay, [kind][kx <= N][tabulated values], from its
// octant [kind][kz <= LZ/2][ky <= N][kx <= N].
template <class C>
__global__ void k_plane_spec(PlaneOrder o, const C* __restrict__ oct, C* __restrict__ out) {
  const int L = o.L, LZ = o.LZ, N = L / 2, n1 = N + 1;
  const long long per = (long long)plane_g_elems(o), total = 2LL * n1 * per;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int kx = (int)((i / per) % n1), kind = (int)(i / per / n1);
    int r = (int)(i % per);
    const int e = r & 1;
    r >>= 1;
    const int ub = o.cw * o.z1, u = r % ub;
    r /= ub;
    const int r2z = LZ / o.z1, k2 = 2 * (r % (r2z / 2)) + e, p = (r / (r2z / 2)) * o.cw + u % o.cw;
    const int ky = p / o.y2 + o.y1 * (p % o.y2), kz = u / o.cw + o.z1 * k2;
    const int fy = ky <= N ? ky : L - ky, fz = kz <= LZ / 2 ? kz : LZ - kz;
    out[i] = oct[(((size_t)kind * (LZ / 2 + 1) + fz) * n1 + fy) * n1 + kx];
  }
}
