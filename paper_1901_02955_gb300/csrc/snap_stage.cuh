// snap_stage.cuh -- device code of one explicit Runge-Kutta stage of the SNAP finite-volume
// scheme (Li & Chen 2019), templated on arithmetic type and field layout. Included by the
// per-configuration translation units kern_*.cu.
//
// One CTA owns a tile of TX x TY x TZ interior cells. It builds the primitives of the tile and
// of a 3-cell halo in each direction in shared memory (ghost cells of the domain boundary are
// synthesised here: mirrored with the normal velocity negated, or wrapped), then for each
// direction reconstructs both face states with WENO5 (Sec. 4.2), solves the LMARS Riemann
// problem (Sec. 4.1) and keeps the face fluxes in shared memory; the owned cells accumulate
// the flux divergence (Eq. forward), add the gravity source, combine the Runge-Kutta stage
// (Sec. 4.3), apply the saturation adjustment (App. D) and store. Face states and fluxes never
// leave the SM.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "snap_internal.h"

namespace snap {

// ------------------------------------------------------------------------------------------
// arithmetic helpers per type
// ------------------------------------------------------------------------------------------
template <class R>
struct Ar;
template <>
struct Ar<float> {
  // a b + c rounded once, whatever the compiler would contract: the same source then rounds
  // the same way in every kernel it is inlined into
  static __device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
  // approximate reciprocal: the special-function unit's rcp.approx.ftz.f32 alone (~1 ulp; a
  // subnormal argument or result flushes to zero, which no reciprocal of the scheme meets:
  // densities, eps + beta >= 1e-6 and the weight sums are normal numbers)
  static __device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
  }
  // a / b as a times the approximate reciprocal (~2 ulp; b a normal number, as every divisor
  // of the scheme is: densities, heat capacities, mixing factors, sound-speed sums)
  static __device__ __forceinline__ float div(float a, float b) { return a * rcp(b); }
  static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
  static __device__ __forceinline__ float exp_(float x) { return expf(x); }
  static __device__ __forceinline__ float log_(float x) { return logf(x); }
  static __device__ __forceinline__ float log1p_(float x) { return log1pf(x); }
  static __device__ __forceinline__ float pow_(float x, float y) { return powf(x, y); }
  // exp2(y log2 x) on the special-function unit: a few ulp when |y log2 x| is small, as for
  // the Exner function (p / 1e5)^(R/c_p) near 1 bar
  static __device__ __forceinline__ float pow_small(float x, float y) { return __powf(x, y); }
  // sqrt of a positive argument as x * rsqrt(x) (~2 ulp): sound speeds
  static __device__ __forceinline__ float sqrt_pos(float x) { return x * rsqrtf(x); }
  // sound speed sqrt(gp / rho) as gp / sqrt(gp rho): one reciprocal square root, no division
  static __device__ __forceinline__ float sound_speed(float gp, float rho) {
    return gp * rsqrtf(gp * rho);
  }
  static constexpr double eps = 1.1920928955078125e-07;
};
template <>
struct Ar<double> {
  static __device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
  // Reciprocal from the hardware's approximate FP64 reciprocal (rcp.approx.ftz.f64, about 1e-6)
  // by one third-order step of the geometric series 1/x = y / (1 - e) = y (1 + e + e^2 + ..),
  // e = 1 - x y: what is left out is e^3 ~ 1e-18, so the result is within an ulp of the IEEE
  // quotient, in three FP64 operations where two Newton-Raphson steps take four (an FP64
  // operation holds its pipe 64 cycles per warp). Zero, infinite, NaN and subnormal x give NaN.
  static __device__ __forceinline__ double rcp(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
  }
  // a / b within about an ulp (the product rounds once more than the quotient)
  static __device__ __forceinline__ double div(double a, double b) { return a * rcp(b); }
  static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
  static __device__ __forceinline__ double exp_(double x) { return exp(x); }
  static __device__ __forceinline__ double log_(double x) { return log(x); }
  static __device__ __forceinline__ double log1p_(double x) { return log1p(x); }
  static __device__ __forceinline__ double pow_(double x, double y) { return pow(x, y); }
  // exp(y log x): the error of the product y log x, |y log x| eps, adds to exp's and log's own
  // few ulp, far below 1e-15 for the Exner function between 0.1 and 10 bar; pow's extended-
  // precision logarithm costs about twice as many FP64 operations
  static __device__ __forceinline__ double pow_small(double x, double y) { return exp(y * log(x)); }
  static __device__ __forceinline__ double sqrt_pos(double x) { return sqrt(x); }
  // gp / sqrt(gp rho) from the approximate reciprocal square root y of x = gp rho (about 1e-6) by
  // one third-order step of the binomial series (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ..,
  // e = 1 - x y^2 (left out: 5 e^3 / 16 ~ 1e-18)
  static __device__ __forceinline__ double sound_speed(double gp, double rho) {
    const double x = gp * rho;
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0), c = gp * y;
    return fma(c * e, fma(0.375, e, 0.5), c);
  }
  static constexpr double eps = 2.220446049250313e-16;
};

// 0 < x < infinity by the bits of x (integer instructions: an FP64 comparison takes an FP64
// pipe slot, 64 cycles of a scheduler)
__device__ __forceinline__ bool finite_positive(double x) {
  return (unsigned)__double2hiint(x) - 1u < 0x7ff00000u - 1u;  // hi word in (0, 0x7ff00000)
}
__device__ __forceinline__ bool finite_positive(float x) {
  return (unsigned)__float_as_int(x) - 1u < 0x7f800000u - 1u;
}

// x > 0 by the bits of x (a NaN may count as positive)
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }

// Field layout of the conserved / primitive vectors (App. B):
// 0 rho_d | 1.. vapours | condensates grouped by vapour | momenta | energy.
template <int NVAP_, int NCOND_, bool D3_>
struct Lay {
  static constexpr int NVAP = NVAP_, NCOND = NCOND_;
  static constexpr bool D3 = D3_;
  static constexpr int NMOM = D3 ? 3 : 2;
  static constexpr int IM0 = 1 + NVAP + NVAP * NCOND;
  static constexpr int NV = IM0 + NMOM + 1;
  static constexpr int IE = NV - 1;
  static __host__ __device__ constexpr int cond(int i, int j) { return 1 + NVAP + i * NCOND + j; }
  // momentum slot of spatial direction d (0 x, 1 y, 2 z)
  static __host__ __device__ constexpr int mom(int d) {
    return D3 ? IM0 + d : IM0 + (d == 2 ? 1 : 0);
  }
  static constexpr bool MOIST = NVAP > 0 && NCOND > 0;
};

template <class R>
__device__ __forceinline__ const CstT<R> &cst(const StageArgs &a);
template <>
__device__ __forceinline__ const CstT<float> &cst<float>(const StageArgs &a) { return a.cf; }
template <>
__device__ __forceinline__ const CstT<double> &cst<double>(const StageArgs &a) { return a.cd; }

// Tile shape: TX x TY x TZ owned cells per CTA of NT threads (TY = 1 in the x-z plane).
// MINB: CTAs per SM the kernel is compiled for (second __launch_bounds__ argument), which caps
// its registers; 0 leaves the register count to the compiler. RESB: the same for the resident step on
// grids of more tiles than SMs (it takes no grid of more tiles than are co-resident).
template <int TX_, int TY_, int TZ_, int NT_ = 256, int MINB_ = 0, int RESB_ = MINB_>
struct TileT {
  static constexpr int TX = TX_, TY = TY_, TZ = TZ_, NT = NT_, MINB = MINB_, RESB = RESB_;
  static constexpr bool MARCH = false;
};
// A tile of TX x TY columns of at most TZ levels (DomDev::cz of them) walked level by level, one
// thread per column (snap_march.cuh).
template <int TX_, int TY_, int TZ_, int MINB_ = 0>
struct MarchT {
  static constexpr int TX = TX_, TY = TY_, TZ = TZ_, NT = TX_ * TY_, MINB = MINB_, RESB = MINB_;
  static constexpr bool MARCH = true;
};

template <class T, bool D3>
struct Box {
  static constexpr int HX = 3, HY = D3 ? 3 : 0, HZ = 3;
  static constexpr int BX = T::TX + 6, BY = T::TY + 2 * HY, BZ = T::TZ + 6;
  static constexpr int NBOX = BX * BY * BZ;
  static constexpr int NFX = (T::TX + 1) * T::TY * T::TZ;
  static constexpr int NFY = D3 ? T::TX * (T::TY + 1) * T::TZ : 0;
  static constexpr int NFZ = T::TX * T::TY * (T::TZ + 1);
  static constexpr int NF = NFX > NFZ ? (NFX > NFY ? NFX : NFY) : (NFZ > NFY ? NFZ : NFY);
  static constexpr int NCELL = T::TX * T::TY * T::TZ;
  static constexpr int CPT = (NCELL + T::NT - 1) / T::NT;  // owned cells per thread
  static __host__ __device__ __forceinline__ int at(int bx, int by, int bz) {
    return (bz * BY + by) * BX + bx;
  }
  // Storage of the primitives in shared memory. x-z: the whole box. 3-D: only the cross the
  // stencils use -- x-lines through the owned y, z range with both x halos (contiguous, so
  // x stencils have unit stride), then the y halos of the owned x, z range, then the z halos
  // of the owned x, y range -- about half the box, which lets a third CTA fit on an SM.
  // Ragged tiles put their far halos inside the owned index range; the fill and the reads use
  // the same map, so a location is never claimed twice.
  static constexpr int NXB = BX * T::TY * T::TZ;
  static constexpr int NYH = D3 ? T::TX * 6 * T::TZ : 0;
  static constexpr int NZH = T::TX * T::TY * 6;
  static constexpr int NSTORE = D3 ? NXB + NYH + NZH : NBOX;
  static __host__ __device__ __forceinline__ int idx(int bx, int by, int bz) {
    if constexpr (!D3) {
      return at(bx, by, bz);
    } else {
      const int oy = by - 3, oz = bz - 3;
      if ((unsigned)oy < (unsigned)T::TY && (unsigned)oz < (unsigned)T::TZ)
        return (oz * T::TY + oy) * BX + bx;
      if ((unsigned)oz < (unsigned)T::TZ)  // y halo: by in 0..2 or TY+3..TY+5
        return NXB + (oz * 6 + (by < 3 ? by : by - T::TY)) * T::TX + (bx - 3);
      return NXB + NYH + ((bz < 3 ? bz : bz - T::TZ) * T::TY + oy) * T::TX + (bx - 3);
    }
  }
  // idx for a location whose z (idx_y) or y (idx_z) lies in the owned range, as along a y or z
  // reconstruction window: one range test instead of two
  static __host__ __device__ __forceinline__ int idx_y(int bx, int by, int bz) {
    const int oy = by - 3, oz = bz - 3;
    if ((unsigned)oy < (unsigned)T::TY) return (oz * T::TY + oy) * BX + bx;
    return NXB + (oz * 6 + (by < 3 ? by : by - T::TY)) * T::TX + (bx - 3);
  }
  static __host__ __device__ __forceinline__ int idx_z(int bx, int by, int bz) {
    const int oy = by - 3, oz = bz - 3;
    if ((unsigned)oz < (unsigned)T::TZ) return (oz * T::TY + oy) * BX + bx;
    return NXB + NYH + ((bz < 3 ? bz : bz - T::TZ) * T::TY + oy) * T::TX + (bx - 3);
  }
};

// Shared-memory arrays of NV fields per location (primitives, face states, fluxes) keep the
// fields of one location together in 16-byte groups (4 floats or 2 doubles), then, for the
// fields left over, an 8-byte pair (floats) and a single field: 11 FP32 fields as 4 + 4 + 2
// + 1, 7 as 4 + 2 + 1, 4 as one group. Each group of an N-location array is a plane of
// N x (group width) values at element N x (its first field), so one vector access moves the
// group of a location: a window point, face state or flux of the four dry fields is one
// 16-byte access instead of four.
template <class R, int NV>
struct SV {
  static constexpr int W = sizeof(R) == 4 ? 4 : 2;       // fields of a 16-byte group
  static constexpr int NF = NV / W;                       // full groups
  static constexpr int T2 = (sizeof(R) == 4 && NV % W >= 2) ? 1 : 0;  // a pair after them
  static constexpr int T1 = (NV % W) % 2;                 // a single last field
  static constexpr int P2 = NF * W;                       // first field of the pair
  static constexpr int P1 = NF * W + 2 * T2;              // the single field
  static_assert(P2 * sizeof(R) % 16 == 0, "the pair's plane must start on a 16-byte boundary");
  static __host__ __device__ __forceinline__ int at(int v, int i, int N) {
    if (v < P2) return ((v / W) * N + i) * W + v % W;
    if (v < P1) return P2 * N + i * 2 + (v - P2);
    return P1 * N + i;
  }
  template <class Vec>
  static __device__ __forceinline__ void ld(const R *p, R *out) {
    const Vec t = *reinterpret_cast<const Vec *>(p);
    const R *e = reinterpret_cast<const R *>(&t);
#pragma unroll
    for (int j = 0; j < int(sizeof(Vec) / sizeof(R)); ++j) out[j] = e[j];
  }
  template <class Vec>
  static __device__ __forceinline__ void st(R *p, const R *in) {
    Vec t;
    R *e = reinterpret_cast<R *>(&t);
#pragma unroll
    for (int j = 0; j < int(sizeof(Vec) / sizeof(R)); ++j) e[j] = in[j];
    *reinterpret_cast<Vec *>(p) = t;
  }
  using V16 = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
  // the fields [first, first + width) of group g of location i (g < NF: a 16-byte group;
  // g == NF: the pair, or the single field)
  static __device__ __forceinline__ void load_group(const R *base, int g, int i, int N, R *out) {
    if (g < NF) {
      ld<V16>(base + (g * N + i) * W, out);
    } else if (T2 && g == NF) {
      ld<float2>(base + P2 * N + i * 2, out);
    } else {
      out[0] = base[P1 * N + i];
    }
  }
  static __device__ __forceinline__ void load(const R *base, int i, int N, R *out) {
#pragma unroll
    for (int g = 0; g < NF; ++g) ld<V16>(base + (g * N + i) * W, out + g * W);
    if constexpr (T2) ld<float2>(base + P2 * N + i * 2, out + P2);
    if constexpr (T1) out[P1] = base[P1 * N + i];
  }
  static __device__ __forceinline__ void store(R *base, int i, int N, const R *in) {
#pragma unroll
    for (int g = 0; g < NF; ++g) st<V16>(base + (g * N + i) * W, in + g * W);
    if constexpr (T2) st<float2>(base + P2 * N + i * 2, in + P2);
    if constexpr (T1) base[P1 * N + i] = in[P1];
  }
};

// What a tile's inner loops read of their domain, copied into shared memory once per tile (the
// descriptor and the profiles in device memory cost two dependent loads per use): levels k0 ..
// k0 + N - 1 of the profiles and the constants, under DomDev's names.
template <class R, int N>
struct Levels {
  R x[N];
  int k0;
  __device__ __forceinline__ R operator[](int k) const { return x[k - k0]; }
  // by one warp
  __device__ __forceinline__ void fill(const R *from, int first, int end, int lane) {
    if (lane == 0) k0 = first;
    for (int i = lane; i < N; i += 32)
      if (first + i >= 0 && first + i < end) x[i] = from[first + i];
  }
};
struct DomSides {
  int bc[6];
  double T_bot;
  __device__ __forceinline__ void fill_sides(const DomDev &D, int lane) {
    if (lane < 6) bc[lane] = D.bc[lane];
    if (lane == 6) T_bot = D.T_bot;
  }
};
// fill: the CTA's first four warps, a profile or two each
template <class R, int N>
struct DomLocal;
template <int N>
struct DomLocal<float, N> : DomSides {
  Levels<float, N> rb_hi, rb_lo, pc_f, pf_f, er_f, er_lo;
  float fidx, fidy, fidz, fgrav;
  __device__ __forceinline__ void fill(const DomDev &D, int first, int tid) {
    const int lane = tid & 31;
    if (tid < 32) {
      fill_sides(D, lane);
      rb_hi.fill(D.rb_hi, first, D.nz, lane);
    } else if (tid < 64) {
      rb_lo.fill(D.rb_lo, first, D.nz, lane);
      pc_f.fill(D.pc_f, first, D.nz, lane);
    } else if (tid < 96) {
      pf_f.fill(D.pf_f, first, D.nz + 1, lane);
      er_f.fill(D.er_f, first, D.nz, lane);
    } else if (tid < 128) {
      er_lo.fill(D.er_lo, first, D.nz, lane);
      if (lane == 0) fidx = D.fidx, fidy = D.fidy, fidz = D.fidz, fgrav = D.fgrav;
    }
  }
};
template <int N>
struct DomLocal<double, N> : DomSides {
  Levels<double, N> rho_bar, p_cell, p_face, e_ref;
  double idx, idy, idz, grav;
  __device__ __forceinline__ void fill(const DomDev &D, int first, int tid) {
    const int lane = tid & 31;
    if (tid < 32) {
      fill_sides(D, lane);
      rho_bar.fill(D.rho_bar, first, D.nz, lane);
    } else if (tid < 64) {
      p_cell.fill(D.p_cell, first, D.nz, lane);
    } else if (tid < 96) {
      p_face.fill(D.p_face, first, D.nz + 1, lane);
    } else if (tid < 128) {
      e_ref.fill(D.e_ref, first, D.nz, lane);
      if (lane == 0) idx = D.idx, idy = D.idy, idz = D.idz, grav = D.grav;
    }
  }
};

// Per-level reference values in the kernel's type: FP32 kernels read FP32 copies, FP64
// kernels the FP64 originals. DD is DomDev, or a kernel's own copy of what it needs of it.
template <class R>
struct Prof;
template <>
struct Prof<float> {
  template <class DD>
  static __device__ __forceinline__ float pc(const DD &D, int k) { return D.pc_f[k]; }
  template <class DD>
  static __device__ __forceinline__ float pf(const DD &D, int k) { return D.pf_f[k]; }
  template <class DD>
  static __device__ __forceinline__ float er(const DD &D, int k) { return D.er_f[k]; }
  // rho - rho_bar_k from the conserved densities y: dry air minus the FP32 head of rho_bar is
  // exact (the two are within a factor of 2), the tracers are added to that small difference,
  // and the FP32 tail of rho_bar (rb_lo) last
  template <class L, class DD>
  static __device__ __forceinline__ float drho(const DD &D, int k, const float *y) {
    float r = y[0] - D.rb_hi[k];
#pragma unroll
    for (int s = 1; s < L::IM0; ++s) r += y[s];
    return r - D.rb_lo[k];
  }
  template <class DD>
  static __device__ __forceinline__ float grav(const DD &D) { return D.fgrav; }
  template <class DD>
  static __device__ __forceinline__ float ih(const DD &D, int d) {
    return d == 0 ? D.fidx : (d == 1 ? D.fidy : D.fidz);
  }
};
template <>
struct Prof<double> {
  template <class DD>
  static __device__ __forceinline__ double pc(const DD &D, int k) { return D.p_cell[k]; }
  template <class DD>
  static __device__ __forceinline__ double pf(const DD &D, int k) { return D.p_face[k]; }
  template <class DD>
  static __device__ __forceinline__ double er(const DD &D, int k) { return D.e_ref[k]; }
  template <class L, class DD>
  static __device__ __forceinline__ double drho(const DD &D, int k, const double *y) {
    double r = y[0];
#pragma unroll
    for (int s = 1; s < L::IM0; ++s) r += y[s];
    return r - D.rho_bar[k];
  }
  template <class DD>
  static __device__ __forceinline__ double grav(const DD &D) { return D.grav; }
  template <class DD>
  static __device__ __forceinline__ double ih(const DD &D, int d) {
    return d == 0 ? D.idx : (d == 1 ? D.idy : D.idz);
  }
};

// ------------------------------------------------------------------------------------------
// thermodynamics (Sec. 2, App. B)
// ------------------------------------------------------------------------------------------
// Conserved -> primitive. y holds the stored state, whose energy entry is rho e - eref with
// eref = pbar / (gamma_d - 1). x receives (rho, q_i, q_ij, u, [v], w, p - pbar), the total
// pressure is returned in p_tot and T in T_out. Dry: p - pbar = (gamma_d - 1)(y_E - K) is
// formed from small numbers. Moist, FP64: the inversion U = rho e - K - A, T = U / C_v, p = R_m T;
// FP32: the same p rewritten as a sum of small numbers.
template <class R, class L, class DD>
__device__ __forceinline__ void cons_to_prim(const Phys &ph, const CstT<R> &C, const DD &D,
                                             int k, const R *y, R *x, R &p_tot, R &T_out) {
  R rho = y[0];
#pragma unroll
  for (int s = 1; s < L::IM0; ++s) rho += y[s];
  const R ir = Ar<R>::rcp(rho);
  x[0] = rho;
#pragma unroll
  for (int s = 1; s < L::IM0; ++s) x[s] = y[s] * ir;
  R K = R(0);
#pragma unroll
  for (int m = 0; m < L::NMOM; ++m) {
    x[L::IM0 + m] = y[L::IM0 + m] * ir;
    K += y[L::IM0 + m] * x[L::IM0 + m];
  }
  K *= R(0.5);
  if constexpr (L::NVAP == 0) {
    // dry: p = (gamma_d - 1) (rho e - K), so p - pbar = (gamma_d - 1) (y_E - K)
    const R pp = C.gm1 * (y[L::IE] - K);
    x[L::IE] = pp;
    const R p = pp + Prof<R>::pc(D, k);
    p_tot = p;
    T_out = p * ir * C.iR_d;
  } else if constexpr (sizeof(R) == 8) {
    // FP64 kernels: U = rho e - K - A, T = U / C_v, p = R_m T directly
    double A = 0.0, Cv = y[0], Rm = y[0];
#pragma unroll
    for (int i = 0; i < L::NVAP; ++i) {
      Cv += ph.sig_v[i] * double(y[1 + i]);
      Rm += ph.inv_eps[i] * double(y[1 + i]);
#pragma unroll
      for (int j = 0; j < L::NCOND; ++j) {
        Cv += ph.sig_c[i][j] * double(y[L::cond(i, j)]);
        A += ph.mu[i][j] * double(y[L::cond(i, j)]);
      }
    }
    Cv *= ph.c_vd;
    Rm *= ph.R_d;
    double U = (double(y[L::IE]) + D.e_ref[k]) - double(K) - A;
    double T = Ar<double>::div(U, Cv);
    double p = Rm * T;
    p_tot = R(p);
    T_out = R(T);
    x[L::IE] = R(p - D.p_cell[k]);
  } else {
    // FP32 kernels: the same p, rewritten so that only small numbers cancel. With the sums
    // over densities C = rho_d + sum sigma_v,i rho_i + sum sigma_ij rho_ij and
    // G = rho_d + sum rho_i / eps_i, p = R_d G T = (gamma_d - 1) (1 + delta) U with
    // delta = (G - C) / C, a sum over tracers only. Since e_ref = pbar / (gamma_d - 1),
    //   p - pbar = (gamma_d - 1) [ (y_E - K - A) + delta (y_E + e_ref - K - A) ],
    // accurate to ~1e-3 Pa at 1e6..1e7 Pa without FP64 (y_E = rho e - e_ref is stored).
    R A = R(0), Cv = y[0], dG = R(0);
#pragma unroll
    for (int i = 0; i < L::NVAP; ++i) {
      Cv += C.sig_v[i] * y[1 + i];
      dG += (C.inv_eps[i] - C.sig_v[i]) * y[1 + i];
#pragma unroll
      for (int j = 0; j < L::NCOND; ++j) {
        Cv += C.sig_c[i][j] * y[L::cond(i, j)];
        dG -= C.sig_c[i][j] * y[L::cond(i, j)];
        A += C.mu[i][j] * y[L::cond(i, j)];
      }
    }
    const R delta = dG * Ar<R>::rcp(Cv);
    const R small = y[L::IE] - K - A;
    const R pp = C.gm1 * (small + delta * (small + Prof<R>::er(D, k)));
    x[L::IE] = pp;
    p_tot = pp + Prof<R>::pc(D, k);
    T_out = R(0);  // not needed by the moist kernels
  }
}

// mixing factors of App. B: num = 1 + sum q_i (sigma_vi - 1) + sum q_ij (sigma_ij - 1),
// den = 1 + sum q_i (1/eps_i - 1) - sum q_ij
template <class R, class L>
__device__ __forceinline__ void mix_factors(const CstT<R> &C, const R *x, R &num, R &den) {
  num = R(1);
  den = R(1);
#pragma unroll
  for (int i = 0; i < L::NVAP; ++i) {
    num += x[1 + i] * C.sigv_m1[i];
    den += x[1 + i] * C.ieps_m1[i];
#pragma unroll
    for (int j = 0; j < L::NCOND; ++j) {
      num += x[L::cond(i, j)] * C.sigc_m1[i][j];
      den -= x[L::cond(i, j)];
    }
  }
}

// ------------------------------------------------------------------------------------------
// LMARS (Sec. 4.1, Eqs. rp, ru) on primitive face states carrying p' = p - pref.
// Operations are what it costs (FP64: 64 pipe cycles of a warp each): sums are kept until their
// factors meet constants, sound speeds take no division, kinetic and latent energy fluxes come from
// the momentum and condensate fluxes. With the shorter FP64 reciprocal and reciprocal square root and
// the same for the viscous flux: density current 1024 x 256 FP64 1.097 -> 1.029 ms per step, FP32
// 39.9 -> 38.6 us; Bryan bubble 200 x 100 FP64 909 -> 869 us.
// rho c from the side averages; upwind side by the sign of u*; flux u* Phi_S + p'* n with
// Phi = (rho_d, rho_i, rho_ij, rho u, [rho v], rho w, rho e + p) of side S.
// ------------------------------------------------------------------------------------------
template <class R, class L>
__device__ __forceinline__ void lmars(const CstT<R> &C, const R *XL, const R *XR, int dir,
                                      R pref, R *F) {
  const int mn = L::mom(dir);
  R numL, denL, numR, denR;
  mix_factors<R, L>(C, XL, numL, denL);
  mix_factors<R, L>(C, XR, numR, denR);
  const R gm1 = C.gm1;
  const R pL = pref + XL[L::IE], pR = pref + XR[L::IE];
  // sound speeds: c^2 = gamma p / rho with gamma = 1 + (gamma_d - 1) den / num (App. B), as
  // (num + (gamma_d - 1) den) p / (num rho): no division
  R cL, cR;
  if constexpr (L::NVAP == 0) {
    cL = Ar<R>::sound_speed(C.gamma_d * pL, XL[0]);
    cR = Ar<R>::sound_speed(C.gamma_d * pR, XR[0]);
  } else {
    cL = Ar<R>::sound_speed(Ar<R>::fma_(gm1, denL, numL) * pL, numL * XL[0]);
    cR = Ar<R>::sound_speed(Ar<R>::fma_(gm1, denR, numR) * pR, numR * XR[0]);
  }
  const R rc4 = (XL[0] + XR[0]) * (cL + cR);  // 4 rho c
  const R uL = XL[mn], uR = XR[mn];
  const R ps = Ar<R>::fma_(R(-0.125) * rc4, uR - uL, R(0.5) * (XL[L::IE] + XR[L::IE]));
  const R us = Ar<R>::fma_(R(-2) * (XR[L::IE] - XL[L::IE]), Ar<R>::rcp(rc4), R(0.5) * (uL + uR));
  const bool left = positive(us);
  R XS[L::NV];
#pragma unroll
  for (int v = 0; v < L::NV; ++v) XS[v] = left ? XL[v] : XR[v];
  const R numS = left ? numL : numR, denS = left ? denL : denR, pS = left ? pL : pR;
  const R mf = us * XS[0];
  R qsum = R(0);
#pragma unroll
  for (int s = 1; s < L::IM0; ++s) {
    F[s] = mf * XS[s];
    qsum += XS[s];
  }
  F[0] = L::IM0 > 1 ? mf * (R(1) - qsum) : mf;
  // energy: u* (rho e + p) = u* p (num / (den (gamma_d - 1)) + 1) + u* (K + A), whose kinetic and
  // latent parts are the momentum and condensate fluxes times u / 2 and mu
  R ka = R(0);
#pragma unroll
  for (int m = 0; m < L::NMOM; ++m) {
    F[L::IM0 + m] = mf * XS[L::IM0 + m];
    ka = Ar<R>::fma_(F[L::IM0 + m], XS[L::IM0 + m], ka);
  }
  F[mn] += ps;
  ka *= R(0.5);
#pragma unroll
  for (int i = 0; i < L::NVAP; ++i)
#pragma unroll
    for (int j = 0; j < L::NCOND; ++j)
      ka = Ar<R>::fma_(C.mu[i][j], F[L::cond(i, j)], ka);
  const R h = L::NVAP == 0 ? C.igm1 + R(1) : Ar<R>::fma_(C.igm1 * numS, Ar<R>::rcp(denS), R(1));
  F[L::IE] = Ar<R>::fma_(us * pS, h, ka);
}

// ------------------------------------------------------------------------------------------
// The temperature inversion's wide numbers: the energy U, the heat capacity, the gas sum and T
// need more digits than FP32 holds (T - T^r decides the saturation pressure, U carries the
// kinetic and latent energies as small differences). FP64 kernels use FP64. FP32 kernels use an
// unevaluated pair h + l of floats (|l| <= ulp(h) / 2, about 48 bits), from the error-free sum
// and product of Knuth and Dekker (the product by a fused multiply-add): on this part an FP64
// instruction holds its pipe 64 cycles per warp, a pair operation is 6 to 12 FP32 instructions.
// A quotient of pairs is good to ~1e-13, where the FP64 form it replaces (one Newton-Raphson
// step) had ~1e-12; sums and products to ~1e-14. Error against FP64 of the adjusted state over
// Jovian and Earth cells: unchanged (below the state's own FP32 rounding).
// ------------------------------------------------------------------------------------------
struct Df {
  float h, l;
};
__device__ __forceinline__ Df quick2(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Df sum2(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Df operator+(Df a, float b) {
  const Df s = sum2(a.h, b);
  return quick2(s.h, __fadd_rn(s.l, a.l));
}
// a + b for |b| <= |a| (the increments of a temperature inversion against its value)
__device__ __forceinline__ Df small_sum(Df a, float b) {
  const Df s = quick2(a.h, b);
  return quick2(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ Df operator+(Df a, Df b) {
  const Df s = sum2(a.h, b.h);
  return quick2(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Df operator-(Df a, Df b) { return a + Df{-b.h, -b.l}; }
__device__ __forceinline__ Df operator*(Df a, float b) {
  const float p = __fmul_rn(a.h, b);
  return quick2(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ Df operator*(Df a, Df b) {
  const float p = __fmul_rn(a.h, b.h);
  return quick2(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p))));
}
// a / b: the approximate quotient q of the heads, then the remainder a - q b over b
__device__ __forceinline__ Df operator/(Df a, Df b) {
  const float r = Ar<float>::rcp(b.h), q = __fmul_rn(a.h, r);
  const float e = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));
  return quick2(q, __fmul_rn(e, r));
}

template <class R>
struct Wide;
template <>
struct Wide<float> {
  using T = Df;
  static __device__ __forceinline__ T of(float x) { return {x, 0.0f}; }
  static __device__ __forceinline__ float r(T x) { return x.h; }
  static __device__ __forceinline__ T diff(float a, float b) { return sum2(a, -b); }
  // a - b to float: the heads' difference is exact within a factor of two, and rounds no more
  // than the result elsewhere
  static __device__ __forceinline__ float gap(T a, T b) {
    return __fadd_rn(__fsub_rn(a.h, b.h), __fsub_rn(a.l, b.l));
  }
  template <class DD>
  static __device__ __forceinline__ T e_ref(const DD &D, int k) { return {D.er_f[k], D.er_lo[k]}; }
  static __device__ __forceinline__ T c_vd(const Phys &, const CstT<float> &C) { return {C.c_vd, C.c_vd_lo}; }
  static __device__ __forceinline__ T R_d(const Phys &, const CstT<float> &C) { return {C.R_d, C.R_d_lo}; }
  static __device__ __forceinline__ T Tref(const Phys &, const CstT<float> &C, int i) { return {C.Tref[i], C.Tref_lo[i]}; }
  static __device__ __forceinline__ T sig_v(const Phys &, const CstT<float> &C, int i) { return {C.sig_v[i], C.sig_v_lo[i]}; }
  static __device__ __forceinline__ T sig_c(const Phys &, const CstT<float> &C, int i, int j) { return {C.sig_c[i][j], C.sig_c_lo[i][j]}; }
  static __device__ __forceinline__ T inv_eps(const Phys &, const CstT<float> &C, int i) { return {C.inv_eps[i], C.inv_eps_lo[i]}; }
  static __device__ __forceinline__ T mu(const Phys &, const CstT<float> &C, int i, int j) { return {C.mu[i][j], C.mu_lo[i][j]}; }
  static __device__ __forceinline__ T quot(T a, T b) { return a / b; }
};
template <>
struct Wide<double> {
  using T = double;
  static __device__ __forceinline__ T of(double x) { return x; }
  static __device__ __forceinline__ double r(T x) { return x; }
  static __device__ __forceinline__ T diff(double a, double b) { return a - b; }
  static __device__ __forceinline__ double gap(T a, T b) { return a - b; }
  template <class DD>
  static __device__ __forceinline__ T e_ref(const DD &D, int k) { return D.e_ref[k]; }
  static __device__ __forceinline__ T c_vd(const Phys &ph, const CstT<double> &) { return ph.c_vd; }
  static __device__ __forceinline__ T R_d(const Phys &ph, const CstT<double> &) { return ph.R_d; }
  static __device__ __forceinline__ T Tref(const Phys &ph, const CstT<double> &, int i) { return ph.Tref[i]; }
  static __device__ __forceinline__ T sig_v(const Phys &ph, const CstT<double> &, int i) { return ph.sig_v[i]; }
  static __device__ __forceinline__ T sig_c(const Phys &ph, const CstT<double> &, int i, int j) { return ph.sig_c[i][j]; }
  static __device__ __forceinline__ T inv_eps(const Phys &ph, const CstT<double> &, int i) { return ph.inv_eps[i]; }
  static __device__ __forceinline__ T mu(const Phys &ph, const CstT<double> &, int i, int j) { return ph.mu[i][j]; }
  static __device__ __forceinline__ T quot(T a, T b) { return Ar<double>::div(a, b); }
};

// T, the heat capacity at constant volume (J/(m^3 K)) and the sum of the gas densities over
// their molar-mass ratios, from the stored conserved values y (energy as rho e - eref): U =
// rho e - K - A, T = U / C_v (Eq. energy, App. B). The FP32 kernels sum the kinetic and latent
// energies and the density they need in FP32: these are up to about 1e-3 of U in clear air and 1e-2 in
// cloud (1e-3 kg/m^3 of water: 2.5e3 of 2e5 J/m^3), so their rounding is 1e-10 to 1e-9 of U, far below
// the 6e-8 of T by which the FP32 state's densities round C_v.
template <class R, class L>
__device__ __forceinline__ void invert_T(const Phys &ph, const CstT<R> &C, const R *y,
                                         typename Wide<R>::T eref, typename Wide<R>::T &T,
                                         typename Wide<R>::T &Cv, typename Wide<R>::T &Rm) {
  using W = Wide<R>;
  Cv = W::of(y[0]);
  Rm = W::of(y[0]);
#pragma unroll
  for (int i = 0; i < L::NVAP; ++i) {
    Cv = Cv + W::sig_v(ph, C, i) * y[1 + i];
    Rm = Rm + W::inv_eps(ph, C, i) * y[1 + i];
#pragma unroll
    for (int j = 0; j < L::NCOND; ++j) Cv = Cv + W::sig_c(ph, C, i, j) * y[L::cond(i, j)];
  }
  R rho = y[0], K2 = R(0), A = R(0);
#pragma unroll
  for (int s = 1; s < L::IM0; ++s) rho += y[s];
#pragma unroll
  for (int m = 0; m < L::NMOM; ++m) K2 = Ar<R>::fma_(y[L::IM0 + m], y[L::IM0 + m], K2);
#pragma unroll
  for (int i = 0; i < L::NVAP; ++i)
#pragma unroll
    for (int j = 0; j < L::NCOND; ++j) A = Ar<R>::fma_(C.mu[i][j], y[L::cond(i, j)], A);
  Cv = Cv * W::c_vd(ph, C);
  if constexpr (sizeof(R) == 4)
    T = W::quot((eref + y[L::IE]) + -(R(0.5) * K2 * Ar<R>::rcp(rho) + A), Cv);
  else
    T = W::quot((eref + y[L::IE]) - R(0.5) * K2 * Ar<R>::rcp(rho) - A, Cv);
}

// ------------------------------------------------------------------------------------------
// App. D saturation adjustment of one cell (isochoric). Each sweep visits the vapours in
// order: projected molar transfer of Eq. dxf with the isochoric alpha, limited to keep both
// phases non-negative, then T and p follow from the conserved energy and the equation of
// state. Returns the sweep count, or -1 without convergence.
// ------------------------------------------------------------------------------------------
// The sweeps of one cell, from the inversion on.
template <class R, class L>
__device__ __forceinline__ int satadj_sweeps(const Phys &ph, const CstT<R> &C, R *y,
                                             typename Wide<R>::T eref, int max_iter) {
  // T from the conserved energy once, in wide numbers (Eq. energy, App. B); after each transfer
  // it is carried forward by the change of the two densities: rho e and the momenta are
  // fixed, so C_v T + A is, and T' = T - (dA + T dC) / (C_v + dC), p' = R_d (R_m + dR_m) T'
  // -- exact algebra, no inversion per sweep. Multiply-adds are explicit fused ones, so that every
  // kernel that inlines this rounds a cell's transfer the same way.
  using W = Wide<R>;
  using A = Ar<R>;
  typename W::T Tw, Cvw, Rw;
  invert_T<R, L>(ph, C, y, eref, Tw, Cvw, Rw);
  Rw = Rw * W::R_d(ph, C);
  R p = W::r(Rw * Tw);
  // the species totals do not change, nor what depends on them alone: the molar sum N and the
  // heat capacity of the mixture. The 3-D layouts (two vapours) form them once; with one vapour,
  // whose cells rarely sweep, the compiler moved them in front of the screen and the 96-domain
  // ensemble slowed from 1.76 to 1.89 ms per step, so there they stay inside the sweep.
  R N, iN, gih;
  const auto mixture = [&]() {
    R heat = R(0);
    N = y[0];
#pragma unroll
    for (int k = 0; k < L::NVAP; ++k) {
      R tot = y[1 + k];
#pragma unroll
      for (int j = 0; j < L::NCOND; ++j) tot += y[L::cond(k, j)];
      N = A::fma_(tot, C.inv_eps[k], N);
      heat = A::fma_(tot * C.inv_eps[k], C.sighat_m1[k], heat);
    }
    iN = A::rcp(N);
    gih = C.gm1 * A::rcp(A::fma_(heat, iN, R(1)));
  };
  if constexpr (L::D3) mixture();
  for (int sweep = 1; sweep <= max_iter; ++sweep) {
    bool conv = true;
#pragma unroll
    for (int i = 0; i < L::NVAP; ++i) {
      if constexpr (!L::D3) mixture();
      R T = W::r(Tw);
      const R dTr = W::gap(Tw, W::Tref(ph, C, i));  // T - T^r kept accurate: s(T) is steep
      R gas = y[0];
#pragma unroll
      for (int k = 0; k < L::NVAP; ++k) gas = A::fma_(y[1 + k], C.inv_eps[k], gas);
      R qv = y[1 + i] * C.inv_eps[i] * iN;
      R qc = y[L::cond(i, 0)] * C.inv_eps[i] * iN;
      R gsum = A::fma_(gas, iN, -qv);
      R t = T * C.inv_Tref[i];
      // p* = p^r exp[beta (1 - 1/t) - delta ln t] with 1 - 1/t = (T - T^r) / T
      const R arg = A::fma_(C.beta[i] * dTr, A::rcp(T), -(C.delta[i] * A::log_(t)));
      R ps = C.pref[i] * Ar<R>::exp_(arg);
      // the arithmetic type holds p* only to ~(|arg| + 2) eps relative (the exponent's own
      // rounding), so the transfer cannot settle below that: the stop test allows 4 times it
      const R tol = fmax(C.satadj_tol, R(4) * (fabs(arg) + R(2)) * R(Ar<R>::eps));
      R s = Ar<R>::div(ps, p);
      R dq;
      if (s >= R(1)) {
        dq = -qc;
      } else {
        R bt = A::fma_(C.beta[i], A::rcp(t), -C.delta[i]);
        R alpha = (bt - R(1)) * gih;
        R om = R(1) - s;
        R r = Ar<R>::div(s, om);
        dq = A::div(A::fma_(-r, gsum, qv),
                    A::fma_(A::div(s, om * om) * bt * alpha, gsum, R(1)));
      }
      R drho;
      if (dq >= qv) {
        dq = qv;
        drho = y[1 + i];
      } else if (dq <= -qc) {
        dq = -qc;
        drho = -y[L::cond(i, 0)];
      } else {
        drho = dq * C.eps[i] * N;
      }
      if (drho != R(0)) {
        const R yv = y[1 + i], yc = y[L::cond(i, 0)];
        y[1 + i] -= drho;
        y[L::cond(i, 0)] += drho;
        // the changes as stored (after rounding to the state's type)
        if constexpr (sizeof(R) == 4) {
          // FP32 states: the increments in FP32 (good to ~1e-7 of themselves, ~1e-10 of T),
          // accumulated into the wide T, heat capacity and gas sum
          const R dv = y[1 + i] - yv, dc = y[L::cond(i, 0)] - yc;
          const R dC = A::fma_(C.sig_v[i], dv, C.sig_c[i][0] * dc) * C.c_vd;
          const R dT = A::fma_(T, dC, C.mu[i][0] * dc) * A::rcp(W::r(Cvw) + dC);
          Tw = small_sum(Tw, -dT);
          Cvw = small_sum(Cvw, dC);
          Rw = small_sum(Rw, C.inv_eps[i] * C.R_d * dv);
        } else {
          const double dv = double(y[1 + i]) - double(yv);
          const double dc = double(y[L::cond(i, 0)]) - double(yc);
          const double dC = (ph.sig_v[i] * dv + ph.sig_c[i][0] * dc) * ph.c_vd;
          Tw -= Ar<double>::div(ph.mu[i][0] * dc + Tw * dC, Cvw + dC);
          Cvw += dC;
          Rw += ph.inv_eps[i] * ph.R_d * dv;
        }
        p = W::r(Rw * Tw);
      }
      if (fabs(dq) > tol * (qv + qc)) conv = false;
    }
    if (conv) return sweep;
  }
  return -1;
}
template <class R, class L>
__device__ __forceinline__ int satadj_cell(const Phys &ph, const CstT<R> &C, R *y, typename Wide<R>::T eref,
                           R eref_r, int max_iter) {
  if constexpr (!L::MOIST) {
    return 0;
  } else {
    if constexpr (sizeof(R) == 4) {
      // FP32 screen: App. D's projected transfer is negative exactly when the vapour's partial
      // pressure is below saturation, and is then limited to the cloud present. A cloud-free
      // vapour that is subsaturated by more than the FP32 error of this estimate (1e-3
      // relative margin) therefore needs no transfer; if all vapours qualify the cell is left
      // unchanged, as the sweeps would leave it.
      R rho = y[0], K2 = R(0), A = R(0), Cv = y[0];
      bool clear = true;
#pragma unroll
      for (int s = 1; s < L::IM0; ++s) rho += y[s];
#pragma unroll
      for (int m = 0; m < L::NMOM; ++m) K2 += y[L::IM0 + m] * y[L::IM0 + m];
#pragma unroll
      for (int i = 0; i < L::NVAP; ++i) {
        Cv += C.sig_v[i] * y[1 + i];
        if (y[L::cond(i, 0)] != R(0)) clear = false;
#pragma unroll
        for (int j = 0; j < L::NCOND; ++j) {
          Cv += C.sig_c[i][j] * y[L::cond(i, j)];
          A += C.mu[i][j] * y[L::cond(i, j)];
        }
      }
      if (clear) {
        // T = U / (c_vd C) with c_vd = R_d / (gamma_d - 1)
        const R T = ((y[L::IE] + eref_r) - R(0.5) * K2 * Ar<R>::rcp(rho) - A) *
                    Ar<R>::rcp(Cv) * C.gm1 * C.iR_d;
#pragma unroll
        for (int i = 0; i < L::NVAP; ++i) {
          const R t = T * C.inv_Tref[i];
          const R ps = C.pref[i] * Ar<R>::exp_(C.beta[i] * (R(1) - Ar<R>::rcp(t)) -
                                               C.delta[i] * Ar<R>::log_(t));
          const R pv = y[1 + i] * C.R_d * C.inv_eps[i] * T;  // rho_i R_i T
          if (!(pv < R(0.999) * ps)) clear = false;
        }
        if (clear) return 1;
      }
    }
    return satadj_sweeps<R, L>(ph, C, y, eref, max_iter);
  }
}

// The cell a ghost at index g (at most n beyond either edge of an axis of n >= 3 cells)
// copies: wrapped on a periodic side (one add or subtract, no integer division), mirrored at a
// wall (flip set).
__device__ __forceinline__ int map_index(int g, int n, int bc_lo, int bc_hi, bool &flip) {
  flip = false;
  if (g < 0) {
    if (bc_lo == 1) return g + n;
    flip = true;
    return -1 - g;
  }
  if (g >= n) {
    if (bc_hi == 1) return g - n;
    flip = true;
    return 2 * n - 1 - g;
  }
  return g;
}

// The domain of a tile: the last whose first tile is not beyond it. Every lane of a warp takes part:
// 32 candidates per round, so two dependent loads for up to 1024 domains (a binary search by
// every thread took log2 of them: 7 for the 96-domain ensemble, before anything else of the tile
// could start).
__device__ __forceinline__ int find_domain(const int *prefix, int ndom, int tile) {
  int lo = 0, n = ndom;  // the answer is one of lo .. lo + n - 1
  while (n > 1) {
    const int step = (n + 31) / 32, i = int(threadIdx.x & 31) * step;
    const bool ok = i < n && __ldg(prefix + lo + i) <= tile;
    const int c = (31 - __clz(__ballot_sync(0xffffffffu, ok))) * step;  // lane 0's test holds
    lo += c;
    n = min(step, n - c);
  }
  return lo;
}

// n / d and n % d for n >= 0 by the precomputed floor(2^32 / d): the high product is the quotient
// or one less
__device__ __forceinline__ void divide(int n, int d, unsigned magic, int &quot, int &rem) {
  quot = int(__umulhi(unsigned(n), magic));
  rem = n - quot * d;
  if (rem >= d) {
    ++quot;
    rem -= d;
  }
}
// Tile coordinates of tile lt of a domain.
__device__ __forceinline__ void tile_coords(const DomDev &D, int lt, int &ix, int &iy, int &iz) {
  int q;
  divide(lt, D.tx, D.tx_magic, q, ix);
  divide(q, D.ty, D.ty_magic, iz, iy);
}

__device__ __forceinline__ double block_max(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (l < int(blockDim.x >> 5)) ? red[l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

// ------------------------------------------------------------------------------------------
// Sedimentation (Sec. 2, Eq. d3 and the momentum and energy equations with terminal
// velocities): condensate (i,j) falling at w^t_j carries through a z face the extra fluxes
// w^t rho_ij (mass), w^t rho_ij u_m (momentum) and w^t rho_ij e_ij with e_ij = c_ij T +
// |u|^2/2 + mu_ij (energy), from the reconstructed state on the side it comes from (above
// when w^t < 0). The frictional heating of the energy equation enters through the total
// mass flux of the gravity-energy source.
// ------------------------------------------------------------------------------------------
template <class R, class L>
__device__ __forceinline__ void sediment_flux(const CstT<R> &C, const R *XL, const R *XR,
                                              R pref, R *F) {
#pragma unroll
  for (int j = 0; j < L::NCOND; ++j) {
    const R wt = C.w_term[j];
    if (wt == R(0)) continue;
    const bool up = wt < R(0);  // falling: the state above the face
    R XS[L::NV];
#pragma unroll
    for (int v = 0; v < L::NV; ++v) XS[v] = up ? XR[v] : XL[v];
    R num, den, u2 = R(0);
    mix_factors<R, L>(C, XS, num, den);
    const R T = (pref + XS[L::IE]) * Ar<R>::rcp(XS[0] * C.R_d * den);
#pragma unroll
    for (int m = 0; m < L::NMOM; ++m) u2 += XS[L::IM0 + m] * XS[L::IM0 + m];
#pragma unroll
    for (int i = 0; i < L::NVAP; ++i) {
      const int c = L::cond(i, j);
      const R ms = wt * XS[0] * XS[c];
      F[c] += ms;
#pragma unroll
      for (int m = 0; m < L::NMOM; ++m) F[L::IM0 + m] += ms * XS[L::IM0 + m];
      F[L::IE] += ms * (C.sig_c[i][j] * C.c_vd * T + R(0.5) * u2 + C.mu[i][j]);
    }
  }
}

// ------------------------------------------------------------------------------------------
// Kessler scheme (Sec. 3) on one cell, backward Euler over dt (Eq. x_n+1), in densities: for
// vapour i with cloud (i,0) and precipitation (i,1), s = rho_v - rho*(T), rho* = p*/(R_i T),
//   saturated (s > 0):  F_v = -k1 s, F_c = k1 s - k3 rho_c rho_r / rho - k2 rho_c,
//                       F_r = k3 rho_c rho_r / rho + k2 rho_c
//   otherwise:          F_v = -k4 rho_r s / rho, F_c = -k3 rho_c rho_r / rho - k2 rho_c,
//                       F_r = k4 rho_r s / rho + k3 rho_c rho_r / rho + k2 rho_c
// (the mass-mixing-ratio rates of Sec. 3 times the fixed total density rho). Newton on
// G = F(y) - (y - y_n)/dt in (rho_v, rho_c) with rho_r = total - rho_v - rho_c, the full
// Jacobian (rho* varies with T, which the reactions change at fixed rho e: dT/drho_k =
// -(mu_k + c_k T)/C_v), one form of the rates at a time: the form of the initial state, then
// the other if the result lies on the wrong side of saturation, else the saturated form.
// T is inverted from the energy in wide numbers. Returns the largest iteration count or -1.
// ------------------------------------------------------------------------------------------
template <class R, class L>
__device__ __forceinline__ void kessler_eval(const Phys &ph, const CstT<R> &C, const R *y,
                                             typename Wide<R>::T T0w, R Cv0, int i, R rho,
                                             const R *yn, R dt,
                                             bool sat, R G[2], R A[2][2], R &s_out,
                                             R &tol_out) {
  const int vi = 1 + i, ci = L::cond(i, 0), ri = L::cond(i, 1);
  // T from T0, the wide temperature of the densities yn this vapour started from, and the
  // phase changes since: rho e and the momenta are fixed, so C_v T + A is (Sec. 2), and
  // T = T0 - (sum_k mu_k d_k + T0 sum_k c_k d_k) / (C_v0 + sum_k c_k d_k) over the vapour,
  // cloud and precipitation changes d_k (the vapour's mu is zero) -- no inversion per
  // Newton iteration
  const R T0 = Wide<R>::r(T0w);
  const R dv = y[vi] - yn[0], dc = y[ci] - yn[1], dr = y[ri] - yn[2];
  const R dC = (C.sig_v[i] * dv + C.sig_c[i][0] * dc + C.sig_c[i][1] * dr) * C.c_vd;
  const R dA = C.mu[i][0] * dc + C.mu[i][1] * dr;
  const R incr = -(dA + T0 * dC) * Ar<R>::rcp(Cv0 + dC);
  const R T = T0 + incr, iT = Ar<R>::rcp(T), t = T * C.inv_Tref[i], it = Ar<R>::rcp(t);
  // T - T^r kept accurate (T0 - T^r from the wide temperature): rho*(T) is steep,
  // d ln rho*/d ln T ~ beta / t ~ 20 near water's triple point, so T rounded to FP32 alone
  // would put ~1e-6 relative noise into s = rho_v - rho* -- the size of the FP32 Newton stop
  // tolerance
  const R dTr = Wide<R>::gap(T0w, Wide<R>::Tref(ph, C, i)) + incr;
  const R arg = C.beta[i] * dTr * iT - C.delta[i] * Ar<R>::log1p_(dTr * C.inv_Tref[i]);
  const R rs = C.pref[i] * Ar<R>::exp_(arg) * C.eps[i] * C.iR_d * iT;  // p* / (R_i T)
  // rho* is held only to ~(|arg| + 2) eps relative: the Newton stop test allows 4 times it
  tol_out = fmax(C.kessler_tol, R(4) * (fabs(arg) + R(2)) * R(Ar<R>::eps));
  const R drs = rs * ((C.beta[i] * it - C.delta[i]) - R(1)) * iT;
  R Cv = y[0];
#pragma unroll
  for (int a = 0; a < L::NVAP; ++a) {
    Cv += C.sig_v[a] * y[1 + a];
#pragma unroll
    for (int b = 0; b < L::NCOND; ++b) Cv += C.sig_c[a][b] * y[L::cond(a, b)];
  }
  const R iCv = Ar<R>::rcp(Cv * C.c_vd);
  // d s / d rho_k for k = vapour, cloud, precipitation (dT/drho_k at fixed energy)
  const R ds[3] = {R(1) + drs * (C.sig_v[i] * C.c_vd * T) * iCv,
                   drs * (C.mu[i][0] + C.sig_c[i][0] * C.c_vd * T) * iCv,
                   drs * (C.mu[i][1] + C.sig_c[i][1] * C.c_vd * T) * iCv};
  const R k1 = C.kk[0], k2 = C.kk[1], k3 = C.kk[2], k4 = C.kk[3], ir = Ar<R>::rcp(rho);
  const R yv = y[vi], yc = y[ci], yr = y[ri], s = yv - rs;
  s_out = s;
  // Equations: the vapour rate G_v and the vapour-plus-cloud rate G_v + G_c, in which the
  // stiff condensation term k1 s cancels exactly (with G_v and G_c separately the 2 x 2
  // determinant would cancel two terms of order k1^2, fatal in FP32 for k1 = 1e9).
  const R acc = k3 * yc * yr * ir;
  R Fv, Fvc, Jv[3], Jvc[3];  // rates and their derivatives by (rho_v, rho_c, rho_r)
  if (sat) {
    Fv = -k1 * s;
    Fvc = -acc - k2 * yc;
#pragma unroll
    for (int q = 0; q < 3; ++q) Jv[q] = -k1 * ds[q];
    Jvc[0] = R(0);
  } else {
    const R e = k4 * yr * ir;
    Fv = -e * s;
    Fvc = -e * s - acc - k2 * yc;
#pragma unroll
    for (int q = 0; q < 3; ++q) Jv[q] = -e * ds[q];
    Jv[2] -= k4 * s * ir;
    Jvc[0] = Jv[0];
  }
  Jvc[1] = (sat ? R(0) : Jv[1]) - k3 * yr * ir - k2;
  Jvc[2] = (sat ? R(0) : Jv[2]) - k3 * yc * ir;
  const R idt = Ar<R>::rcp(dt);
  G[0] = Fv - (yv - yn[0]) * idt;
  G[1] = Fvc - ((yv - yn[0]) + (yc - yn[1])) * idt;
  // 2 x 2 Jacobian in (rho_v, rho_c) with rho_r = total - rho_v - rho_c
  A[0][0] = Jv[0] - Jv[2] - idt;
  A[0][1] = Jv[1] - Jv[2];
  A[1][0] = Jvc[0] - Jvc[2] - idt;
  A[1][1] = Jvc[1] - Jvc[2] - idt;
}

template <class R, class L>
__device__ __forceinline__ int kessler_branch(const Phys &ph, const CstT<R> &C, R *y,
                                              typename Wide<R>::T T0, R Cv0, int i, R rho,
                                              const R *yn,
                                              R tot, R dt, bool sat, R &s) {
  const int vi = 1 + i, ci = L::cond(i, 0), ri = L::cond(i, 1);
  y[vi] = yn[0];
  y[ci] = yn[1];
  y[ri] = yn[2];
  for (int m = 1; m <= ph.kessler_max_iter; ++m) {
    R G[2], A[2][2], tol;
    kessler_eval<R, L>(ph, C, y, T0, Cv0, i, rho, yn, dt, sat, G, A, s, tol);
    const R idet = Ar<R>::rcp(A[0][0] * A[1][1] - A[0][1] * A[1][0]);
    const R dv = (-G[0] * A[1][1] + G[1] * A[0][1]) * idet;
    const R dc = (-G[1] * A[0][0] + G[0] * A[1][0]) * idet;
    y[vi] += dv;
    y[ci] += dc;
    y[ri] = tot - y[vi] - y[ci];
    if (fabs(dv) + fabs(dc) <= tol * (fabs(y[vi]) + fabs(y[ci]) + fabs(y[ri]))) {
      R Gt[2], At[2][2], tt;
      kessler_eval<R, L>(ph, C, y, T0, Cv0, i, rho, yn, dt, sat, Gt, At, s, tt);
      return m;
    }
  }
  return -1;
}

template <class R, class L>
__device__ int kessler_cell(const Phys &ph, const CstT<R> &C, R *y, typename Wide<R>::T eref,
                            R dt) {
  if constexpr (!(L::NVAP > 0 && L::NCOND >= 2)) {
    return 0;
  } else {
    R rho = R(0);
#pragma unroll
    for (int s = 0; s < L::IM0; ++s) rho += y[s];
    // the cell's temperature and heat capacity once in wide numbers; each vapour then updates
    // them by its own phase changes
    using W = Wide<R>;
    typename W::T T0, Cv0, Rm0;
    invert_T<R, L>(ph, C, y, eref, T0, Cv0, Rm0);
    int worst = 0;
    for (int i = 0; i < L::NVAP; ++i) {
      const int vi = 1 + i, ci = L::cond(i, 0), ri = L::cond(i, 1);
      const R yn[3] = {y[vi], y[ci], y[ri]};
      const R tot = yn[0] + yn[1] + yn[2];
      R G[2], A[2][2], s0, s, tol0;
      const R cv0 = W::r(Cv0);
      kessler_eval<R, L>(ph, C, y, T0, cv0, i, rho, yn, dt, true, G, A, s0, tol0);
      const bool first = s0 > R(0);
      int it = kessler_branch<R, L>(ph, C, y, T0, cv0, i, rho, yn, tot, dt, first, s);
      if (!(it > 0 && (first ? s > R(0) : s <= R(0)))) {
        it = kessler_branch<R, L>(ph, C, y, T0, cv0, i, rho, yn, tot, dt, !first, s);
        if (!(it > 0 && (!first ? s > R(0) : s <= R(0))))
          it = kessler_branch<R, L>(ph, C, y, T0, cv0, i, rho, yn, tot, dt, true, s);
      }
      {  // this vapour's phase changes, in wide numbers, carried to the next vapour's T0 and C_v0
        const typename W::T dv = W::diff(y[vi], yn[0]), dc = W::diff(y[ci], yn[1]);
        const typename W::T dr = W::diff(y[ri], yn[2]);
        const typename W::T dC = (W::sig_v(ph, C, i) * dv + W::sig_c(ph, C, i, 0) * dc +
                                  W::sig_c(ph, C, i, 1) * dr) * W::c_vd(ph, C);
        const typename W::T dA = W::mu(ph, C, i, 0) * dc + W::mu(ph, C, i, 1) * dr;
        T0 = T0 - W::quot(dA + T0 * dC, Cv0 + dC);
        Cv0 = Cv0 + dC;
      }
      if (it < 0)
        worst = -1;
      else if (worst >= 0 && it > worst)
        worst = it;
    }
    return worst;
  }
}

__device__ __forceinline__ float block_max_f(float v, float *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (l < int(blockDim.x >> 5)) ? red[l] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

// Asynchronous global -> shared copy of one element (cp.async, completed by cp_async_wait):
// the stage input Y^n of the owned cells is fetched while the tile is being computed.
template <class R>
__device__ __forceinline__ void cp_async_elem(R *smem_dst, const R *gmem_src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  if constexpr (sizeof(R) == 4)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem_src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem_src) : "memory");
}
// Flag accesses of the resident step: a load with acquire and a store with release
// semantics at device scope (the data written before the release is visible to a CTA whose
// acquire load saw the flag).
__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int *p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned int *p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ------------------------------------------------------------------------------------------
// the fused stage kernel
// ------------------------------------------------------------------------------------------
// WENO5 of Sec. 4.2 evaluated once per cell c for both of its faces from the five cells
// (a, b, c, d, e) = Q_{c-2} .. Q_{c+2}:
//   qm = left state at face c+1/2   = I_weno(Q_{c-2}, .., Q_{c+2})
//   qp = right state at face c-1/2  = I_weno(Q_{c+2}, .., Q_{c-2})  (Eq. q+, mirror stencil)
// The Jiang-Shu smoothness indicator of a 3-cell triple does not depend on the direction the
// triple is read in, so the three indicators (and their inverse squares) serve both faces; the
// mirror stencil takes them in reverse order. The linear weights are folded into the
// candidate coefficients, so each face needs one normalising reciprocal.
// Common factors cancel in a face's normalisation sum_k w_k q_k / sum_k w_k, so the kernel
// takes (a) every eps + beta_k times 12/13: beta_k = 13/12 s^2 + 1/4 r^2 becomes s^2 + 3/13 r^2
// against eps 12/13; (b) the linear weights (0.1, 0.6, 0.3) times 10: each normalisation
// g0 + 6 g1 + 3 g2 is two fused multiply-adds. And since the weights sum to the normalisation,
// a face state is its middle candidate q_1 plus what the outer two add to it,
//   q = q_1 + [w_0 (q_0 - q_1) + w_2 (q_2 - q_1)] / sum_k w_k,
// where the departures are third differences of the window: with the neighbour differences
// w = b - a, u = c - b, v = d - c, z = e - d, the second differences s0 = u - w, s1 = v - u,
// s2 = z - v (which the indicators need anyway) and D1 = s1 - s0, D2 = s2 - s1,
//   left state at c+1/2:  q_1 = c + (u + 2 v) / 6, q_0 - q_1 = -D1 / 3, q_2 - q_1 = -D2 / 6;
//   right state at c-1/2: q_1 = c - (v + 2 u) / 6, q_0 - q_1 = D2 / 3, q_2 - q_1 = D1 / 6
// (the mirror stencil turns (w, u, v, z) into (-z, -v, -u, -w), which swaps D1 and D2 with a
// sign). The two bracketed sums share the products g0 D1 and g2 D2. Against the weighted sum
// of the three offsets q_k - c this form takes 38 instead of 48 operations per window, and the
// weights' rounding only reaches the third-difference term. Measured: density current 1024 x
// 256, FP32 41.9 -> 39.9 us and FP64 1.203 -> 1.097 ms per step; the 96-domain ensemble 1.88 ->
// 1.81 ms per step.
template <class R>
__device__ __forceinline__ void weno5_pair(R a, R b, R c, R d, R e, R eps, R &qm, R &qp) {
  // every multiply-add below is an explicit fused one (Ar::fma_), so that each kernel
  // instantiation rounds the same way whatever its register allocation
  using A = Ar<R>;
  constexpr R k3 = R(3.0 / 13.0);
  // (w, z, s2 and r2 with the opposite signs)
  const R u = c - b, v = d - c, w = a - b, z = d - e;
  const R s0 = u + w, s1 = v - u, s2 = v + z;
  const R r0 = A::fma_(R(3), u, w);  // a - 4b + 3c
  const R r1 = u + v;                // d - b
  const R r2 = A::fma_(R(3), v, z);  // -(3c - 4d + e)
  eps *= R(12.0 / 13.0);
  const R e0 = A::fma_(k3 * r0, r0, A::fma_(s0, s0, eps));
  const R e1 = A::fma_(k3 * r1, r1, A::fma_(s1, s1, eps));
  const R e2 = A::fma_(k3 * r2, r2, A::fma_(s2, s2, eps));
  // inverse squares 1 / (eps + beta_k)^2, shared by both faces. FP64 (whose reciprocal is a
  // multi-instruction sequence on a slow pipe) forms them up to the common factor
  // 1 / (e0 e1 e2)^2, which cancels in each face's normalisation: g_k = (product of the other
  // two e)^2 -- no reciprocal here, and the two normalisations below share one.
  R g0, g1, g2;
  if constexpr (sizeof(R) == 8) {
    g0 = e1 * e2;
    g1 = e0 * e2;
    g2 = e0 * e1;
  } else {
    g0 = A::rcp(e0);
    g1 = A::rcp(e1);
    g2 = A::rcp(e2);
  }
  g0 *= g0;
  g1 *= g1;
  g2 *= g2;
  const R Sm = A::fma_(R(3), g2, A::fma_(R(6), g1, g0));
  const R Sp = A::fma_(R(3), g0, A::fma_(R(6), g1, g2));
  // the bracketed sums, -(g0 D1 / 3 + g2 D2 / 2) and g0 D1 / 2 + g2 D2 / 3, from the halves of
  // the third differences (signs chosen so that no operand needs a negation, which the packed
  // instructions of weno5_pair2 do not have, and few constants, which take them a register pair each)
  const R h1 = R(0.5) * s1;
  const R P = g0 * A::fma_(R(-0.5), s0, h1);  // g0 D1 / 2
  const R Q = g2 * A::fma_(R(0.5), s2, h1);   // -g2 D2 / 2
  const R Nm = A::fma_(R(-2.0 / 3.0), P, Q);
  const R Np = A::fma_(R(-2.0 / 3.0), Q, P);
  const R cm = A::fma_(R(1.0 / 6.0), r1 + v, c);
  const R cp = A::fma_(R(-0.5), r1, cm);  // c - (v + 2 u) / 6
  if constexpr (sizeof(R) == 8) {
    // 1/Sm = Sp / (Sm Sp) and 1/Sp = Sm / (Sm Sp); one division each only if the product
    // leaves the exponent range (g ~ e^4, so Sm Sp ~ e^8: eps far below 1e-6 or huge beta)
    const R Z = A::rcp(Sm * Sp);  // NaN outside the normal range: the test below fails
    if (finite_positive(Z)) {
      qm = A::fma_(Nm, Sp * Z, cm);
      qp = A::fma_(Np, Sm * Z, cp);
    } else {
      qm = cm + Nm / Sm;
      qp = cp + Np / Sp;
    }
  } else {
    qm = A::fma_(Nm, A::rcp(Sm), cm);
    qp = A::fma_(Np, A::rcp(Sp), cp);
  }
}

// weno5_pair<float> for two variables at once on the packed FP32x2 pipe of sm_100-class SMs
// (one instruction per two lanes of arithmetic: the reconstruction is issue-bound); the
// reciprocals stay scalar on the special-function unit.
__device__ __forceinline__ float2 f2c(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 f2rcp(float2 x) {
  return make_float2(Ar<float>::rcp(x.x), Ar<float>::rcp(x.y));
}
__device__ __forceinline__ void weno5_pair2(float2 a, float2 b, float2 c, float2 d, float2 e,
                                            float eps, float2 &qm, float2 &qp) {
  // the operations of weno5_pair in the same order (differences as fused multiply-adds by -1,
  // which round the same)
  const float2 k3 = f2c(3.0f / 13.0f), m1f = f2c(-1.0f);
  const float2 u = __ffma2_rn(m1f, b, c), v = __ffma2_rn(m1f, c, d), w = __ffma2_rn(m1f, b, a),
               z = __ffma2_rn(m1f, e, d);
  const float2 s0 = __fadd2_rn(u, w), s1 = __ffma2_rn(m1f, u, v), s2 = __fadd2_rn(v, z);
  const float2 r0 = __ffma2_rn(f2c(3.0f), u, w);
  const float2 r1 = __fadd2_rn(u, v);
  const float2 r2 = __ffma2_rn(f2c(3.0f), v, z);
  const float2 ke = f2c(eps * (12.0f / 13.0f));
  const float2 e0 = __ffma2_rn(__fmul2_rn(k3, r0), r0, __ffma2_rn(s0, s0, ke));
  const float2 e1 = __ffma2_rn(__fmul2_rn(k3, r1), r1, __ffma2_rn(s1, s1, ke));
  const float2 e2 = __ffma2_rn(__fmul2_rn(k3, r2), r2, __ffma2_rn(s2, s2, ke));
  float2 g0 = f2rcp(e0), g1 = f2rcp(e1), g2 = f2rcp(e2);
  g0 = __fmul2_rn(g0, g0);
  g1 = __fmul2_rn(g1, g1);
  g2 = __fmul2_rn(g2, g2);
  const float2 Sm = __ffma2_rn(f2c(3.0f), g2, __ffma2_rn(f2c(6.0f), g1, g0));
  const float2 Sp = __ffma2_rn(f2c(3.0f), g0, __ffma2_rn(f2c(6.0f), g1, g2));
  const float2 h1 = __fmul2_rn(f2c(0.5f), s1);
  const float2 P = __fmul2_rn(g0, __ffma2_rn(f2c(-0.5f), s0, h1));
  const float2 Q = __fmul2_rn(g2, __ffma2_rn(f2c(0.5f), s2, h1));
  const float2 Nm = __ffma2_rn(f2c(-2.0f / 3.0f), P, Q);
  const float2 Np = __ffma2_rn(f2c(-2.0f / 3.0f), Q, P);
  const float2 cm = __ffma2_rn(f2c(1.0f / 6.0f), __fadd2_rn(r1, v), c);
  const float2 cp = __ffma2_rn(f2c(-0.5f), r1, cm);
  qm = __ffma2_rn(Nm, f2rcp(Sm), cm);
  qp = __ffma2_rn(Np, f2rcp(Sp), cp);
}

// CFL rate sum_d (|u_d| + c) / dx_d in the kernel's type (FP32 kernels: FP32; the time step
// only needs a few digits). The energy entry is stored as rho e - eref.
template <class R, class L>
__device__ __forceinline__ R cell_rate_r(const CstT<R> &C, const R *y, R eref, R idx, R idy,
                                         R idz) {
  R rho = y[0];
#pragma unroll
  for (int s = 1; s < L::IM0; ++s) rho += y[s];
  const R ir = Ar<R>::rcp(rho);
  R K2 = R(0);
#pragma unroll
  for (int m = 0; m < L::NMOM; ++m) K2 += y[L::IM0 + m] * y[L::IM0 + m];
  R num = R(1), den = R(1), A = R(0), Cv = y[0], Rm = y[0];
#pragma unroll
  for (int i = 0; i < L::NVAP; ++i) {
    num += y[1 + i] * ir * C.sigv_m1[i];
    den += y[1 + i] * ir * C.ieps_m1[i];
    Cv += C.sig_v[i] * y[1 + i];
    Rm += C.inv_eps[i] * y[1 + i];
#pragma unroll
    for (int j = 0; j < L::NCOND; ++j) {
      num += y[L::cond(i, j)] * ir * C.sigc_m1[i][j];
      den -= y[L::cond(i, j)] * ir;
      Cv += C.sig_c[i][j] * y[L::cond(i, j)];
      A += C.mu[i][j] * y[L::cond(i, j)];
    }
  }
  const R U = (y[L::IE] + eref) - R(0.5) * K2 * ir - A;
  // p = R_d R_m T and T = U / (c_vd C_v), with R_m, C_v here the sums over densities
  const R p = C.gm1 * Rm * Ar<R>::div(U, Cv);
  const R gam = R(1) + C.gm1 * Ar<R>::div(den, num);
  const R c = Ar<R>::sqrt_pos(gam * p * ir);
  R r = (fabs(y[L::mom(0)]) * ir + c) * idx + (fabs(y[L::mom(2)]) * ir + c) * idz;
  if constexpr (L::D3) r += (fabs(y[L::mom(1)]) * ir + c) * idy;
  return r;
}

template <class R, class L, bool VISC, class T>
struct StageSmem {
  using B = Box<T, L::D3>;
  static constexpr size_t prim = (sizeof(R) * L::NV * B::NSTORE + 15) / 16 * 16;
  static constexpr size_t visc = VISC ? (sizeof(R) * 2 * B::NSTORE + 15) / 16 * 16 : 0;
  // left states (then fluxes) and right states, each array starting on a 16-byte boundary:
  // the grouped layout moves 16-byte vectors
  static constexpr size_t face_half = (sizeof(R) * L::NV * B::NF + 15) / 16 * 16;
  static constexpr size_t face = 2 * face_half;
  static constexpr size_t red = 32 * sizeof(double);
  static constexpr size_t base = prim + visc + face + red;
  static_assert(prim % 16 == 0 && visc % 16 == 0 && face_half % 16 == 0 && red % 16 == 0,
                "every shared-memory array of the stage starts on a 16-byte boundary");
  // Y^n of the owned cells, prefetched by cp.async, when it costs no resident CTA per SM
  // (228 KB of shared memory per SM, 1 KB reserved per CTA)
  static constexpr size_t yn_bytes = sizeof(R) * L::NV * B::NCELL;
  static constexpr bool PREFETCH = 233472 / (base + yn_bytes + 1024) >= 233472 / (base + 1024);
  static constexpr size_t yn = PREFETCH ? yn_bytes : 0;
  static constexpr size_t total = base + yn;
};

// Grid-wide barrier of the persistent step kernel (all CTAs co-resident by a cooperative
// launch). Every wait is bounded: after spin_limit clock cycles (about 2 s by default) the CTA
// records kFlagTimeout and proceeds, so a fault can corrupt results but never hang the device.
// The host clears the barrier state before every persistent launch, so a count left behind by
// a wait that gave up does not open a later barrier early. absent_cta (a test aid, -1 in
// normal use) names a CTA that neither arrives nor waits, which makes every other CTA's wait
// run out.
__device__ __forceinline__ void grid_barrier(GridSync *gs, unsigned int nblocks,
                                             unsigned int *flags, long long spin_limit,
                                             int absent_cta) {
  __syncthreads();
  if (threadIdx.x == 0 && int(blockIdx.x) != absent_cta) {
    volatile unsigned int *vgen = &gs->gen;
    const unsigned int g = *vgen;
    __threadfence();
    const unsigned int arrived = atomicAdd(&gs->count, 1u);
    if (arrived == nblocks - 1) {
      atomicExch(&gs->count, 0u);
      __threadfence();
      atomicAdd(&gs->gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == g) {
        if (clock64() - t0 > spin_limit) {
          atomicOr(flags, (unsigned)kFlagTimeout);
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// The stage's time step (one thread per CTA). The first tile of a domain records it in stage 0 and
// clears the domain's CFL maximum in stage 1; kept is the CTA's own stage-0 time step (resident
// step, stages 1 and 2).
template <bool RES>
__device__ __forceinline__ double stage_dt(const StageArgs &a, const DomDev &D, int stage, int lt,
                                           double kept) {
  if (stage == 0) {
    const double dt = a.dt_override > 0.0 ? a.dt_override
                      : (D.dt_fixed > 0.0 ? D.dt_fixed
                                          : D.cfl / __longlong_as_double((long long)*D.rate));
    if (lt == 0) *D.dt_step = dt;
    return dt;
  }
  if (RES) return kept;
  if (stage == 1 && lt == 0) *D.rate = 0ull;
  return *(volatile double *)D.dt_step;
}

// Where the cell (gx, gy, gz) beyond a tile along direction dirn (it may lie outside the domain, at
// most 3 cells) takes its values from: the interior cell itself, a slab neighbour's cell, or for
// a ghost of the domain boundary the cell it wraps to or mirrors (flip). Field v is src[v * stride].
template <class R>
struct HaloCell {
  const R *src;
  long long stride;
  int side;  // the domain side along dirn that a ghost lies beyond (x-, x+, y-, y+, z-, z+)
  int gz;    // level of the source cell
  bool flip;
};
template <class R>
__device__ __forceinline__ HaloCell<R> halo_cell(const StageArgs &a, const DomDev &D, int stage,
                                                 const R *Ys, int gx, int gy, int gz, int dirn) {
  HaloCell<R> h;
  const int nx = D.nx, ny = D.ny, nz = D.nz;
  h.side = 2 * dirn + ((dirn == 0 ? gx : (dirn == 1 ? gy : gz)) < 0 ? 0 : 1);
  h.flip = false;
  if (dirn == 0 && (gx < 0 || gx >= nx) && D.bc[h.side] == kBcHalo && !a.buf_s) {
    // a slab boundary: the neighbouring slab's cells (a linked domain's stage input, or the
    // ghost buffer the caller filled)
    const int s = h.side, hn = D.hnx[s];
    h.stride = (long long)hn * ny * nz;
    h.src = reinterpret_cast<const R *>(D.hsrc[s][stage]) + ((long long)gz * ny + gy) * hn +
            D.hoff[s] + (s ? gx - nx : gx + 3);
  } else {
    if (dirn == 0) gx = map_index(gx, nx, D.bc[0], D.bc[1], h.flip);
    if (dirn == 1) gy = map_index(gy, ny, D.bc[2], D.bc[3], h.flip);
    if (dirn == 2) gz = map_index(gz, nz, D.bc[4], D.bc[5], h.flip);
    h.stride = D.ncell;
    h.src = Ys + (((long long)gz * ny + gy) * nx + gx);
  }
  h.gz = gz;
  return h;
}
// Its conserved values; CG reads past L1 (cells other CTAs wrote during this launch).
template <class R, int NV, bool CG>
__device__ __forceinline__ void load_fields(const R *src, long long stride, R *y) {
#pragma unroll
  for (int v = 0; v < NV; ++v) y[v] = CG ? __ldcg(src + v * stride) : src[v * stride];
}
// Its primitives from those values: a wall's ghost has the normal velocity, or at a no-slip wall
// every component, negated, and below a fixed-temperature floor the temperature T_bot.
template <class R, class L, class DD>
__device__ __forceinline__ void halo_prim(const DD &D, const Phys &ph, const CstT<R> &C,
                                          const HaloCell<R> &h, int dirn, const R *y, R *x, R &pt) {
  R Tt;
  cons_to_prim<R, L>(ph, C, D, h.gz, y, x, pt, Tt);
  if (h.flip) {
    // (selects, not x[mom(dirn)]: a run-time index would put x into local memory)
    const bool all = D.bc[h.side] == kBcNoSlip;
#pragma unroll
    for (int m = L::IM0; m < L::IM0 + L::NMOM; ++m)
      if (all || m == L::mom(dirn)) x[m] = -x[m];
    // Sec. 6 lower boundary: the ghost holds T_bot at the mirrored pressure and composition,
    // so its density is p / (R_d den T_bot) (App. B: p = rho R_d den T, den the mixing
    // factor), the mirrored density times T / T_bot
    if (h.side == 4 && D.T_bot > 0.0) {
      R num, den;
      mix_factors<R, L>(C, x, num, den);
      x[0] = pt * C.iR_d * Ar<R>::rcp(den * R(D.T_bot));
    }
  }
}

// Both face states of the cell whose five-cell window is at locations o of the grouped array
// base (N locations): one group of fields at a time (the group's five window points, one vector
// access each); FP32 pairs on the packed FP32x2 pipe, an odd field alone.
template <class R, int NV>
__device__ __forceinline__ void recon_window(const R *base, const int (&o)[5], int N, R weps,
                                             R *QM, R *QP) {
  using V = SV<R, NV>;
#pragma unroll
  for (int g = 0; g < V::NF + V::T2 + V::T1; ++g) {
    const int f0 = g < V::NF ? g * V::W : (g == V::NF && V::T2 ? V::P2 : V::P1);
    const int n = g < V::NF ? V::W : (g == V::NF && V::T2 ? 2 : 1);
    R X[5][V::W];
#pragma unroll
    for (int k = 0; k < 5; ++k) V::load_group(base, g, o[k], N, X[k]);
    if constexpr (sizeof(R) == 4) {
#pragma unroll
      for (int j = 0; j + 1 < V::W; j += 2) {
        if (j + 1 < n) {
          float2 qm, qp;
          weno5_pair2(make_float2(X[0][j], X[0][j + 1]), make_float2(X[1][j], X[1][j + 1]),
                      make_float2(X[2][j], X[2][j + 1]), make_float2(X[3][j], X[3][j + 1]),
                      make_float2(X[4][j], X[4][j + 1]), weps, qm, qp);
          QM[f0 + j] = qm.x, QM[f0 + j + 1] = qm.y, QP[f0 + j] = qp.x, QP[f0 + j + 1] = qp.y;
        }
      }
      if (n == 1)
        weno5_pair<R>(X[0][0], X[1][0], X[2][0], X[3][0], X[4][0], weps, QM[f0], QP[f0]);
    } else {
#pragma unroll
      for (int j = 0; j < V::W; ++j)
        if (j < n)
          weno5_pair<R>(X[0][j], X[1][j], X[2][j], X[3][j], X[4][j], weps, QM[f0 + j], QP[f0 + j]);
    }
  }
}

// The end of a cell's stage: gravity and forcing added to the flux divergence acc, the stage
// combine, saturation adjustment, microphysics (stage 2) and the checks of the result yo. ys is
// the stage input, yn(v) field v of Y^n (stages 1 and 2), mb and mt the total-mass fluxes
// through the cell's lower and upper z faces.
template <class R, class L, bool MICRO, class DD, class YN>
__device__ __forceinline__ void finish_cell(const StageArgs &a, const DD &D, const Phys &ph,
                                            const CstT<R> &C, int stage, R dt, int k, const R *ys,
                                            R *acc, R mb, R mt, YN yn, R *yo) {
  using P = Prof<R>;
  const R grav = P::grav(D);
  // vertical momentum: -(rho - rho_bar) g (Eq. mom3 with the reference balance removed)
  acc[L::mom(2)] -= P::template drho<L>(D, k, ys) * grav;
  // energy: -g (F_rho,k-1/2 + F_rho,k+1/2) / 2 with the vertical total-mass fluxes
  acc[L::IE] -= grav * R(0.5) * (mb + mt);
  if constexpr (MICRO && L::MOIST) {
    // forcing of the Jovian simulation (Sec. 6) by the level's reference pressure
    const R pk = P::pc(D, k);
    if (C.cool_rate != R(0) && pk >= C.cool_p_lo && pk <= C.cool_p_hi) {
      R Cv = ys[0];  // heat capacity at constant volume / c_vd
#pragma unroll
      for (int i2 = 0; i2 < L::NVAP; ++i2) {
        Cv += C.sig_v[i2] * ys[1 + i2];
#pragma unroll
        for (int j2 = 0; j2 < L::NCOND; ++j2) Cv += C.sig_c[i2][j2] * ys[L::cond(i2, j2)];
      }
      acc[L::IE] -= Cv * C.c_vd * C.cool_rate;
    }
    if (C.sponge_itau0 != R(0) && pk * C.sponge_ip0 < R(1)) {
      const R r = pk * C.sponge_ip0, rate = C.sponge_itau0 * Ar<R>::rcp(r * r);
      acc[L::mom(0)] -= ys[L::mom(0)] * rate;
      if constexpr (L::D3) acc[L::mom(1)] -= ys[L::mom(1)] * rate;
    }
  }
#pragma unroll
  for (int v = 0; v < L::NV; ++v) {
    const R s1 = ys[v] + dt * acc[v];
    if (stage == 0) {
      yo[v] = s1;
    } else {
      // (1 - w) Y^n + w s1 as Y^n + w (s1 - Y^n): the two weights sum to exactly one. With 1/3
      // and 2/3 each rounded to FP32 they sum to 1 + 3e-8, which scales the whole state by that
      // much every step (a mass drift of 1e-3 over 30,000 steps). An explicit fused
      // multiply-add, so that every kernel that inlines this rounds it the same way.
      const R y0 = yn(v), wgt = stage == 1 ? R(0.25) : R(2.0 / 3.0);
      yo[v] = fma(wgt, s1 - y0, y0);
    }
  }
  if constexpr (L::MOIST) {
    if (ph.satadj) {
      const int it = satadj_cell<R, L>(ph, C, yo, Wide<R>::e_ref(D, k), P::er(D, k),
                                          ph.satadj_max_iter);
      if (it < 0)
        atomicOr(a.flags, (unsigned)kFlagNoConv);
      else if (it > 2)
        atomicMax(a.max_sweeps, it);
    }
    // the microphysics follows each step (time splitting), over the step's dt
    if (MICRO && stage == 2 && ph.kessler) {
      if (kessler_cell<R, L>(ph, C, yo, Wide<R>::e_ref(D, k), dt) < 0)
        atomicOr(a.flags, (unsigned)kFlagNoConv);
    }
  }
  R rs = R(0);
#pragma unroll
  for (int s = 0; s < L::IM0; ++s) rs += yo[s];
  if (!(rs > R(0)) || !isfinite(yo[L::IE])) atomicOr(a.flags, (unsigned)kFlagNonFinite);
}

// Viscous flux of one face (Sec. 5.1), added to F: -rho_f nu du/dn and -rho_f nu (u_f du/dn + c_pd
// Pi_f dtheta/dn) between the cells at locations bl and br, with the face means as halves of
// sums: k = rho_f nu / dn. ih: inverse cell size along the face's normal.
template <class R, class L>
__device__ __forceinline__ void viscous_flux(const CstT<R> &C, R ih, const R *prim, const R *th,
                                             const R *pi, int bl, int br, int N, R *F) {
  using V = SV<R, L::NV>;
  R XL[L::NV], XR[L::NV];
  V::load(prim, bl, N, XL);
  V::load(prim, br, N, XR);
  const R k = (XL[0] + XR[0]) * (R(0.5) * C.nu * ih);
  R w2 = (C.c_pd * (pi[bl] + pi[br])) * (th[br] - th[bl]);
#pragma unroll
  for (int m = L::IM0; m < L::IM0 + L::NMOM; ++m) {
    const R du = XR[m] - XL[m];
    F[m] = Ar<R>::fma_(-k, du, F[m]);
    w2 = Ar<R>::fma_(XL[m] + XR[m], du, w2);
  }
  F[L::IE] = Ar<R>::fma_(R(-0.5) * k, w2, F[L::IE]);
}

// One stage over the CTA's 3-D one-shot tiles. RES (the resident step, one tile per CTA for all three
// stages): for stages 1 and 2 ys holds the owned cells' stage input on entry (the previous
// stage's output, kept in registers) instead of being loaded; Y^n of the owned cells is kept
// in shared memory from stage 0 on; the time step of stage 0 stays in s_red[0]; ghost cells
// are read past L1 (other CTAs wrote them during this launch); the CFL maximum goes to
// D.rate_next (the step's own rate stays readable until every CTA has formed its time step);
// ys receives the stage output.
template <class R, class L, bool VISC, class T, bool MICRO, bool RES = false>
__device__ __forceinline__ void stage_tiles(const StageArgs &a, const int stage,
                                            unsigned char *smem,
                                            R (&ys)[Box<T, L::D3>::CPT][L::NV]) {
  static_assert(L::D3, "the x-z plane has its own kernel (plane_tiles)");
  using B = Box<T, L::D3>;
  using S = StageSmem<R, L, VISC, T>;
  using P = Prof<R>;
  constexpr int NV = L::NV;
  constexpr int TX = T::TX, TY = T::TY, TZ = T::TZ, NT = T::NT;
  R *s_prim = reinterpret_cast<R *>(smem);
  R *s_th = reinterpret_cast<R *>(smem + S::prim);
  R *s_pi = s_th + (VISC ? B::NSTORE : 0);
  R *s_fl = reinterpret_cast<R *>(smem + S::prim + S::visc);  // left states, then fluxes
  R *s_fr = s_fl + S::face_half / sizeof(R);                   // right states
  using V = SV<R, NV>;
  double *s_red = reinterpret_cast<double *>(smem + S::prim + S::visc + S::face);
  R *s_yn = reinterpret_cast<R *>(smem + S::base);  // used when S::PREFETCH
  const Phys &ph = a.ph;
  const CstT<R> &C = cst<R>(a);
  const R weps = C.weno_eps;
  const int tid = threadIdx.x;

  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int dm = find_domain(a.tile_domain, a.ndom, tile);
    const DomDev &D = a.doms[dm];
    const int nx = D.nx, ny = D.ny, nz = D.nz;
    const long long ncell = D.ncell;
    const int lt = tile - D.tile_begin;
    int ix, iy, iz;
    tile_coords(D, lt, ix, iy, iz);
    const int x0 = ix * TX, y0 = iy * TY, z0 = iz * TZ;
    const int ex = min(TX, nx - x0), ey = min(TY, ny - y0), ez = min(TZ, nz - z0);
    const R *Ys = reinterpret_cast<const R *>(a.buf_s ? a.buf_s : D.buf[stage]);
    const R *Yn = reinterpret_cast<const R *>(a.buf_n ? a.buf_n : D.buf[0]);
    R *Yo = reinterpret_cast<R *>(a.buf_o ? a.buf_o : D.buf[stage == 0 ? 1 : (stage == 1 ? 2 : 0)]);
    // the stage's time step, formed once per CTA
    if (tid == 0) s_red[0] = stage_dt<RES>(a, D, stage, lt, s_red[0]);

    // ---- 1. owned cells: load, keep the conserved values, store primitives -------------
    if constexpr (S::PREFETCH && !RES) {
      if (stage != 0) {
#pragma unroll
        for (int m = 0; m < B::CPT; ++m) {
          const int c = tid + m * NT;
          const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
          if (c < B::NCELL && lx < ex && ly < ey && lz < ez) {
            const long long g = ((long long)(z0 + lz) * ny + (y0 + ly)) * nx + (x0 + lx);
#pragma unroll
            for (int v = 0; v < NV; ++v) cp_async_elem<R>(s_yn + v * B::NCELL + c, Yn + v * ncell + g);
          }
        }
        cp_async_commit();
      }
    }
#pragma unroll
    for (int m = 0; m < B::CPT; ++m) {
      const int c = tid + m * NT;
      const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
      if (c < B::NCELL && lx < ex && ly < ey && lz < ez && (!RES || stage == 0)) {
        const long long g = ((long long)(z0 + lz) * ny + (y0 + ly)) * nx + (x0 + lx);
#pragma unroll
        for (int v = 0; v < NV; ++v) ys[m][v] = Ys[v * ncell + g];
      }
    }
    // halo item h of the cross (x, y, z): its place in the box, direction and layer
    constexpr int NHX = 6 * TY * TZ, NHY = 6 * TX * TZ, NHZ = 6 * TX * TY, NH = NHX + NHY + NHZ;
    auto halo_item = [&](int h, int &bx, int &by, int &bz, int &dirn, int &layer) {
      if (h < NHX) {
        const int r = h % 6, q = h / 6, ly = q % TY, lz = q / TY;
        layer = r;
        bx = r < 3 ? r : ex + r;
        by = ly + B::HY;
        bz = lz + 3;
        dirn = 0;
        return ly < ey && lz < ez;
      }
      if (h < NHX + NHY) {
        const int hh = h - NHX, lx = hh % TX, r = (hh / TX) % 6, lz = hh / (6 * TX);
        layer = r;
        bx = lx + 3;
        by = r < 3 ? r : ey + r;
        bz = lz + 3;
        dirn = 1;
        return lx < ex && lz < ez;
      }
      const int hh = h - NHX - NHY, lx = hh % TX, ly = (hh / TX) % TY, r = hh / (TX * TY);
      layer = r;
      bx = lx + 3;
      by = ly + B::HY;
      bz = r < 3 ? r : ez + r;
      dirn = 2;
      return h < NH && lx < ex && ly < ey;
    };
    // The dry FP32 layout has registers for the thread's halo items: their loads go out together with
    // the owned cells', before any conversion. Waited for one after the other they were what a small
    // grid waits for most: 39 x 25 x 15 cells 30.8 -> 28.7 us per step (resident 37.1 -> 34.7), 48 x
    // 48 x 48 53.6 -> 51.0, 64 x 64 x 64 99.9 -> 94.4; the moist FP32 layout has 80 registers a thread,
    // and FP64 is bound by its pipe.
    constexpr int NE = (NH + NT - 1) / NT;
    constexpr bool EARLY = sizeof(R) == 4 && NV * NE <= 25;
    HaloCell<R> he[EARLY ? NE : 1];
    R yh[EARLY ? NE : 1][NV];
    int hb[EARLY ? NE : 1], hl[EARLY ? NE : 1];  // box location (-1: none), direction and layer
    if constexpr (EARLY) {
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        int bx, by, bz, dirn, layer;
        const bool ok = halo_item(tid + e * NT, bx, by, bz, dirn, layer);
        hb[e] = -1;
        if (ok) {
          hb[e] = B::idx(bx, by, bz);
          hl[e] = dirn | layer << 2;
          he[e] = halo_cell<R>(a, D, stage, Ys, x0 + bx - 3, y0 + by - B::HY, z0 + bz - 3, dirn);
          load_fields<R, NV, RES>(he[e].src, he[e].stride, yh[e]);
        }
      }
    }
#pragma unroll
    for (int m = 0; m < B::CPT; ++m) {
      const int c = tid + m * NT;
      const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
      if (c < B::NCELL && lx < ex && ly < ey && lz < ez) {
        const int k = z0 + lz;
        if constexpr (RES && S::PREFETCH) {
          if (stage == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) s_yn[v * B::NCELL + c] = ys[m][v];
          }
        }
        R x[NV], pt, Tt;
        cons_to_prim<R, L>(ph, C, D, k, ys[m], x, pt, Tt);
        const int bi = B::idx(lx + 3, ly + B::HY, lz + 3);
        V::store(s_prim, bi, B::NSTORE, x);
        if constexpr (VISC) {
          const R Pi = Ar<R>::pow_small(pt * R(1e-5), C.kappa);
          s_th[bi] = pt * Ar<R>::rcp(x[0] * Pi) * C.iR_d;
          s_pi[bi] = Pi;
        }
      }
    }
    // ---- 2. halo of the cross, boundary ghosts synthesised ------------------------------
    auto store_halo = [&](const HaloCell<R> &hc, const R *y, int bi, int dirn, int layer) {
      R x[NV], pt;
      halo_prim<R, L>(D, ph, C, hc, dirn, y, x, pt);
      V::store(s_prim, bi, B::NSTORE, x);
      // the viscous heat flux reads theta and the Exner function only on the two sides of
      // a face, so of the halo only the ring next to the tile (layers 2 and 3) needs them
      if constexpr (VISC) {
        if (layer == 2 || layer == 3) {
          const R Pi = Ar<R>::pow_small(pt * R(1e-5), C.kappa);
          s_th[bi] = pt * Ar<R>::rcp(x[0] * Pi) * C.iR_d;
          s_pi[bi] = Pi;
        }
      }
    };
    if constexpr (EARLY) {
#pragma unroll
      for (int e = 0; e < NE; ++e)
        if (hb[e] >= 0) store_halo(he[e], yh[e], hb[e], hl[e] & 3, hl[e] >> 2);
    } else {
      for (int h = tid; h < NH; h += NT) {
        int bx, by, bz, dirn, layer;
        if (!halo_item(h, bx, by, bz, dirn, layer)) continue;
        const HaloCell<R> hc =
            halo_cell<R>(a, D, stage, Ys, x0 + bx - 3, y0 + by - B::HY, z0 + bz - 3, dirn);
        R y[NV];
        load_fields<R, NV, RES>(hc.src, hc.stride, y);
        store_halo(hc, y, B::idx(bx, by, bz), dirn, layer);
      }
    }
    __syncthreads();
    const R dt = R(s_red[0]);

    R acc[B::CPT][NV];
#pragma unroll
    for (int m = 0; m < B::CPT; ++m)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[m][v] = R(0);

    // ---- 3. per direction: WENO5 per cell (both faces), LMARS per face, divergence -------
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int fx = d == 0, fy = d == 1, fz = d == 2;
      // face array strides: faces along d are numbered 0..T_d
      const int sx = TX + fx, sy = TY + fy;
      const int ed = d == 0 ? ex : (d == 1 ? ey : ez);
      // 3a. reconstruction over the owned cells and one more on each side along d
      {
        const int rx = TX + 2 * fx, ry = TY + 2 * fy, rz = TZ + 2 * fz;
        const int nrec = rx * ry * rz;
        constexpr int MAXREC = (TX + 2) * (TY + 2) * (TZ + 2);
#pragma unroll
        for (int r = 0; r < (MAXREC + NT - 1) / NT; ++r) {
          const int it = tid + r * NT;
          int lx = it % rx, ly = (it / rx) % ry, lz = it / (rx * ry);
          lx -= fx;
          ly -= fy;
          lz -= fz;
          const int ld = fx ? lx : (fy ? ly : lz);
          if (it < nrec && ld <= ed && lx < ex + fx && ly < ey + fy && lz < ez + fz) {
            // the five cells of the window along d: unit stride along the x-lines, mapped one by
            // one where a y or z window leaves them
            int o[5];
            if (!fx) {
              // the window's fixed coordinate lies in the owned range
#pragma unroll
              for (int k = 0; k < 5; ++k)
                o[k] = fy ? B::idx_y(lx + 3, ly + B::HY + (k - 2), lz + 3)
                          : B::idx_z(lx + 3, ly + B::HY, lz + 3 + (k - 2));
            } else {
              const int bi = B::idx(lx + 3, ly + B::HY, lz + 3);
#pragma unroll
              for (int k = 0; k < 5; ++k) o[k] = bi + k - 2;
            }
            const int fl = ((lz + fz) * sy + (ly + fy)) * sx + (lx + fx);  // face c+1/2
            const int fr = (lz * sy + ly) * sx + lx;                        // face c-1/2
            const bool has_l = ld < ed, has_r = ld >= 0;
            R QM[NV], QP[NV];
            recon_window<R, NV>(s_prim, o, B::NSTORE, weps, QM, QP);
            if (has_l) V::store(s_fl, fl, B::NF, QM);
            if (has_r) V::store(s_fr, fr, B::NF, QP);
          }
        }
      }
      __syncthreads();
      // 3b. LMARS flux per face (and the viscous flux), written over the left state
      {
        const int nface = sx * sy * (TZ + fz);
#pragma unroll
        for (int r = 0; r < (B::NF + NT - 1) / NT; ++r) {
          const int f = tid + r * NT;
          const int ix = f % sx, iy = (f / sx) % sy, iz = f / (sx * sy);
          if (f >= nface || ix >= ex + fx || iy >= ey + fy || iz >= ez + fz) continue;
          R QL[NV], QR[NV], F[NV];
          V::load(s_fl, f, B::NF, QL);
          V::load(s_fr, f, B::NF, QR);
          const R pref = fz ? P::pf(D, z0 + iz) : P::pc(D, z0 + iz);
          lmars<R, L>(C, QL, QR, d, pref, F);
          if constexpr (L::MOIST && MICRO) {
            // no condensate passes a wall (both z sides are)
            const int kf = z0 + iz;
            if (fz && ph.sediment && kf != 0 && kf != nz) sediment_flux<R, L>(C, QL, QR, pref, F);
          }
          if constexpr (VISC) {
            const int bi = B::idx(ix + 3, iy + B::HY, iz + 3);  // right cell of the face
            const int bl = B::idx(ix + 3 - fx, iy + B::HY - fy, iz + 3 - fz);
            viscous_flux<R, L>(C, P::ih(D, d), s_prim, s_th, s_pi, bl, bi, B::NSTORE, F);
          }
          V::store(s_fl, f, B::NF, F);
        }
      }
      __syncthreads();
      // 3c. flux divergence of the owned cells (Eq. forward)
      const R ih = P::ih(D, d);
#pragma unroll
      for (int m = 0; m < B::CPT; ++m) {
        const int c = tid + m * NT;
        const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
        if (c < B::NCELL && lx < ex && ly < ey && lz < ez) {
          const int f0 = (lz * sy + ly) * sx + lx;
          const int f1 = ((lz + fz) * sy + (ly + fy)) * sx + (lx + fx);
          R F1[NV], F0[NV];
          V::load(s_fl, f1, B::NF, F1);
          V::load(s_fl, f0, B::NF, F0);
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[m][v] -= (F1[v] - F0[v]) * ih;
        }
      }
      if (d != 2) __syncthreads();
    }

    // ---- 4. gravity source, stage combine, saturation adjustment, store ------------------
    if constexpr (S::PREFETCH && !RES) {
      if (stage != 0) cp_async_wait();  // this thread's own copies of Y^n
    }
    R rate_max = R(0);
#pragma unroll
    for (int m = 0; m < B::CPT; ++m) {
      const int c = tid + m * NT;
      const int lx = c % TX, ly = (c / TX) % TY, lz = c / (TX * TY);
      if (c < B::NCELL && lx < ex && ly < ey && lz < ez) {
        const int k = z0 + lz;
        // vertical total-mass fluxes through the cell's two z faces
        const int f0 = (lz * TY + ly) * TX + lx;
        const int f1 = ((lz + 1) * TY + ly) * TX + lx;
        R mb = R(0), mt = R(0);
#pragma unroll
        for (int s = 0; s < L::IM0; ++s) {
          mb += s_fl[V::at(s, f0, B::NF)];
          mt += s_fl[V::at(s, f1, B::NF)];
        }
        const long long g = ((long long)k * ny + (y0 + ly)) * nx + (x0 + lx);
        R yo[NV];
        finish_cell<R, L, MICRO>(
            a, D, ph, C, stage, dt, k, ys[m], acc[m], mb, mt,
            [&](int v) { return S::PREFETCH ? s_yn[v * B::NCELL + c] : Yn[v * ncell + g]; }, yo);
#pragma unroll
        for (int v = 0; v < NV; ++v) Yo[v * ncell + g] = yo[v];
        if constexpr (RES) {
#pragma unroll
          for (int v = 0; v < NV; ++v) ys[m][v] = yo[v];
        }
        if (stage == 2)
          rate_max = fmax(rate_max, cell_rate_r<R, L>(C, yo, P::er(D, k), P::ih(D, 0),
                                                      P::ih(D, 1), P::ih(D, 2)));
      }
    }
    if (stage == 2) {
      double bm;
      if constexpr (sizeof(R) == 4)
        bm = double(block_max_f(rate_max, reinterpret_cast<float *>(s_red + 1)));
      else
        bm = block_max(rate_max, s_red + 1);
      if (tid == 0)
        atomicMax(RES ? D.rate_next : D.rate, (unsigned long long)__double_as_longlong(bm));
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// the x-z plane
// ------------------------------------------------------------------------------------------
// Shared memory of an x-z tile: the boxed primitives (and theta, Exner function), per direction
// the left states of its faces, overwritten by their fluxes, the right states of the far x
// faces, the local copy of the domain, and Y^n of the owned cells where that costs no resident
// CTA (228 KB of shared memory per SM, 1 KB reserved per CTA).
template <class R, class L, bool VISC, class T>
struct PlaneSmem {
  using B = Box<T, false>;
  static constexpr int RPB = T::NT / T::TX;                     // rows per round of the CTA
  static constexpr int M = (T::TZ + 2 + RPB - 1) / RPB;         // rounds over rows -1 .. TZ
  static constexpr int NX = (T::TX + 1) * T::TZ, NZ = T::TX * (T::TZ + 1);
  static constexpr int NEXTRA = 4 * T::TX + 6 * T::TZ;          // halo cells outside those rows
  static constexpr size_t bytes(int n, int nv) { return (sizeof(R) * nv * n + 15) / 16 * 16; }
  static constexpr size_t visc_off = bytes(B::NBOX, L::NV);
  static constexpr size_t x_off = visc_off + (VISC ? bytes(B::NBOX, 2) : 0);
  static constexpr size_t z_off = x_off + bytes(NX, L::NV);
  static constexpr size_t r_off = z_off + bytes(NZ, L::NV);
  static constexpr size_t red_off = r_off + bytes(T::TZ, L::NV);
  static constexpr size_t dom_off = red_off + 32 * sizeof(double);
  using Dom = DomLocal<R, T::TZ + 7>;  // levels z0 - 3 .. z0 + TZ + 3
  // both directions in the same phases (three barriers instead of five) where their states fit
  // the registers: the four dry fields (5 % of the FP32 step), not the seven moist ones
  static constexpr bool BOTH = L::NV <= 4;
  static constexpr size_t base = dom_off + (sizeof(Dom) + 15) / 16 * 16;
  static constexpr size_t yn_bytes = sizeof(R) * L::NV * T::NT * M;
  static constexpr bool PREFETCH = 233472 / (base + yn_bytes + 1024) >= 233472 / (base + 1024);
  static constexpr size_t total = base + (PREFETCH ? yn_bytes : 0);
};

// One stage over the CTA's x-z tiles. A thread keeps column lx = tid mod TX of rows row, row + RPB,
// .. (row -1 and row ez are the z halo next to the tile, reconstructed for the outer z faces): it
// converts these cells, reconstructs them, solves the face on their lower side from its own right
// state (kept in registers) and its neighbour's left state (shared memory), and finishes them
// with its own lower flux and the neighbour's. Rounds, rows and columns are powers of two or
// constants, so an item's locations are the thread's plus an immediate. RES as for stage_tiles.
//
// Bound by instruction issue (FP32) and the FP64 pipe (FP64). All loads of a tile go out together,
// then the domain's profiles, then the conversions; dividing item numbers into rows and columns,
// reading the profiles through the descriptor and exchanging both states of every face through
// shared memory took 911 instructions per cell where this takes 826 (density current 1024 x 256,
// FP32: 38.6 -> 35.8 us per step; 96-domain ensemble 1.83 -> 1.74 ms, one moist bubble of 61 x 47
// cells 31.9 -> 29 us). Four cells per thread instead of two at the same tile are slower (39.5
// us; ensemble 2.16 ms): the warps are what hides the phases' latency.
template <class R, class L, bool VISC, class T, bool MICRO, bool RES = false>
__device__ __forceinline__ void plane_tiles(const StageArgs &a, const int stage,
                                            unsigned char *smem,
                                            R (&ys)[PlaneSmem<R, L, VISC, T>::M][L::NV]) {
  using S = PlaneSmem<R, L, VISC, T>;
  using B = Box<T, false>;
  using P = Prof<R>;
  using V = SV<R, L::NV>;
  constexpr int NV = L::NV, TX = T::TX, TZ = T::TZ, NT = T::NT, M = S::M, RPB = S::RPB;
  constexpr int BX = B::BX, NB = B::NBOX, NE = (S::NEXTRA + NT - 1) / NT;
  static_assert((TX & (TX - 1)) == 0 && NT % TX == 0 && 2 * TZ <= NT && NT >= 128, "columns of whole rounds");
  R *s_prim = reinterpret_cast<R *>(smem);
  R *s_th = reinterpret_cast<R *>(smem + S::visc_off), *s_pi = s_th + (VISC ? NB : 0);
  R *s_x = reinterpret_cast<R *>(smem + S::x_off), *s_z = reinterpret_cast<R *>(smem + S::z_off);
  R *s_r = reinterpret_cast<R *>(smem + S::r_off);
  double *s_red = reinterpret_cast<double *>(smem + S::red_off);
  R *s_dt = reinterpret_cast<R *>(s_red + 31);
  typename S::Dom &Dl = *reinterpret_cast<typename S::Dom *>(smem + S::dom_off);
  R *s_yn = reinterpret_cast<R *>(smem + S::base);  // used when S::PREFETCH
  const Phys &ph = a.ph;
  const CstT<R> &C = cst<R>(a);
  const R weps = C.weno_eps;
  const int tid = threadIdx.x, lx = tid % TX, row = tid / TX;
  const int bi0 = (row + 2) * BX + lx + 3;  // the thread's cell of round 0 (row row - 1)

  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    const int dm = find_domain(a.tile_domain, a.ndom, tile);
    const DomDev &D = a.doms[dm];
    const int nx = D.nx, nz = D.nz;
    const long long ncell = D.ncell;
    const int lt = tile - D.tile_begin;
    int ix, iz;
    divide(lt, D.tx, D.tx_magic, iz, ix);
    const int cz = D.cz;  // rows per tile, at most TZ
    const int x0 = ix * TX, z0 = iz * cz;
    const int ex = min(TX, nx - x0), ez = min(cz, nz - z0);
    const R *Ys = reinterpret_cast<const R *>(a.buf_s ? a.buf_s : D.buf[stage]);
    const R *Yn = reinterpret_cast<const R *>(a.buf_n ? a.buf_n : D.buf[0]);
    R *Yo = reinterpret_cast<R *>(a.buf_o ? a.buf_o : D.buf[stage == 0 ? 1 : (stage == 1 ? 2 : 0)]);
    auto level = [&](int r) {  // row r's level, mirrored at the z walls
      const int k = z0 + r;
      return k < 0 ? -1 - k : (k >= nz ? 2 * nz - 1 - k : k);
    };
    auto owned = [&](int m) { return lx < ex && (unsigned)(row + m * RPB - 1) < (unsigned)ez; };
    // ---- 1. every load of the tile, then the local copy of the domain, then the conversions
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int r = row + m * RPB - 1;
      if (lx < ex && r <= ez && !(RES && stage > 0 && owned(m)))
        load_fields<R, NV, RES>(Ys + ((long long)level(r) * nx + (x0 + lx)), ncell, ys[m]);
    }
    // the halo cells outside rows -1 .. ez: four z rows, then three columns on each x side
    HaloCell<R> hc[NE];
    R yh[NE][NV];
    int hb[NE];  // box location, -1: none
    bool hx[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int h = tid + e * NT;
      hb[e] = -1;
      hx[e] = h >= 4 * TX;
      int x = 0, r = 0;
      bool ok = false;
      if (!hx[e]) {
        const int q = h / TX;
        x = h % TX;
        r = q < 2 ? q - 3 : ez + q - 1;
        ok = x < ex;
      } else if (h < S::NEXTRA) {
        const int q = (h - 4 * TX) % 6;
        r = (h - 4 * TX) / 6;
        x = q < 3 ? q - 3 : ex + q - 3;
        ok = r < ez;
      }
      if (ok) {
        hb[e] = (r + 3) * BX + x + 3;
        if (hx[e])
          hc[e] = halo_cell<R>(a, D, stage, Ys, x0 + x, 0, z0 + r, 0);
        else
          hc[e] = halo_cell<R>(a, D, stage, Ys, x0 + x, 0, z0 + r, 2);
        load_fields<R, NV, RES>(hc[e].src, hc[e].stride, yh[e]);
      }
    }
    if constexpr (S::PREFETCH && !RES) {
      if (stage != 0) {
#pragma unroll
        for (int m = 0; m < M; ++m)
          if (owned(m)) {
            const R *src = Yn + ((long long)(z0 + row + m * RPB - 1) * nx + (x0 + lx));
#pragma unroll
            for (int v = 0; v < NV; ++v)
              cp_async_elem<R>(s_yn + (m * NV + v) * NT + tid, src + v * ncell);
          }
        cp_async_commit();
      }
    }
    Dl.fill(D, z0 - 3, tid);
    if (tid == NT - 1) {  // while the tile's loads are on their way
      const double dt = stage_dt<RES>(a, D, stage, lt, s_red[0]);
      s_red[0] = dt;
      *s_dt = R(dt);
    }
    __syncthreads();
    auto store_prim = [&](const R *x, R pt, int b, bool heat) {
      V::store(s_prim, b, NB, x);
      // the viscous heat flux reads theta and the Exner function only on the two sides of a
      // face: not beyond the ring next to the tile
      if constexpr (VISC) {
        if (heat) {
          const R Pi = Ar<R>::pow_small(pt * R(1e-5), C.kappa);
          s_th[b] = pt * Ar<R>::rcp(x[0] * Pi) * C.iR_d;
          s_pi[b] = Pi;
        }
      }
    };
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int r = row + m * RPB - 1;
      if (lx < ex && r <= ez) {
        HaloCell<R> c;
        c.gz = level(r);
        c.flip = c.gz != z0 + r;
        c.side = z0 + r < 0 ? 4 : 5;
        R x[NV], pt;
        halo_prim<R, L>(Dl, ph, C, c, 2, ys[m], x, pt);
        store_prim(x, pt, bi0 + m * RPB * BX, true);
        if constexpr (RES && S::PREFETCH) {
          if (stage == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) s_yn[(m * NV + v) * NT + tid] = ys[m][v];
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < NE; ++e)
      if (hb[e] >= 0) {
        R x[NV], pt;
        halo_prim<R, L>(Dl, ph, C, hc[e], hx[e] ? 0 : 2, yh[e], x, pt);
        const int q = (tid + e * NT - 4 * TX) % 6;
        store_prim(x, pt, hb[e], hx[e] && (q == 2 || q == 3));
      }
    __syncthreads();

    // ---- 2. per direction: states, face fluxes (over the left states), divergence. Qx, Qz: the
    // right state of the cell's lower face, then that face's flux. x: the owned cells, and the
    // column on either side by the threads whose last row lies above the tile
    R acc[M][NV], Q[S::BOTH ? 2 : 1][M][NV];
    auto &Qx = Q[0], &Qz = Q[S::BOTH ? 1 : 0];
    const int e = NT - 1 - tid;  // the last threads first
    auto x_states = [&]() {
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (owned(m)) {
          const int r = row + m * RPB - 1, b = bi0 + m * RPB * BX;
          const int o[5] = {b - 2, b - 1, b, b + 1, b + 2};
          R QM[NV];
          recon_window<R, NV>(s_prim, o, NB, weps, QM, Qx[m]);
          V::store(s_x, r * (TX + 1) + lx + 1, S::NX, QM);
        }
      if (e < 2 * TZ) {
        const int r = e >> 1;
        const bool far = e & 1;
        if (r < ez) {
          const int b = (r + 3) * BX + (far ? ex : -1) + 3;
          const int o[5] = {b - 2, b - 1, b, b + 1, b + 2};
          R QM[NV], QP[NV];
          recon_window<R, NV>(s_prim, o, NB, weps, QM, QP);
          if (far)
            V::store(s_r, r, TZ, QP);
          else
            V::store(s_x, r * (TX + 1), S::NX, QM);
        }
      }
    };
    auto x_fluxes = [&]() {
#pragma unroll
      for (int m = 0; m < M; ++m)
        if (owned(m)) {
          const int r = row + m * RPB - 1, f = r * (TX + 1) + lx, b = bi0 + m * RPB * BX;
          R QL[NV], F[NV];
          V::load(s_x, f, S::NX, QL);
          lmars<R, L>(C, QL, Qx[m], 0, P::pc(Dl, z0 + r), F);
          if constexpr (VISC)
            viscous_flux<R, L>(C, P::ih(Dl, 0), s_prim, s_th, s_pi, b - 1, b, NB, F);
          V::store(s_x, f, S::NX, F);
#pragma unroll
          for (int v = 0; v < NV; ++v) Qx[m][v] = F[v];
        }
      if (e < TZ && e < ez) {
        const int f = e * (TX + 1) + ex, b = (e + 3) * BX + ex + 3;
        R QL[NV], QR[NV], F[NV];
        V::load(s_x, f, S::NX, QL);
        V::load(s_r, e, TZ, QR);
        lmars<R, L>(C, QL, QR, 0, P::pc(Dl, z0 + e), F);
        if constexpr (VISC)
          viscous_flux<R, L>(C, P::ih(Dl, 0), s_prim, s_th, s_pi, b - 1, b, NB, F);
        V::store(s_x, f, S::NX, F);
      }
    };
    auto x_divergence = [&](int m) {
      if (owned(m)) {
        R F1[NV];
        V::load(s_x, (row + m * RPB - 1) * (TX + 1) + lx + 1, S::NX, F1);
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[m][v] = -((F1[v] - Qx[m][v]) * P::ih(Dl, 0));
      }
    };
    auto z_states = [&](int m) {
      const int r = row + m * RPB - 1, b = bi0 + m * RPB * BX;
      if (lx < ex && r <= ez) {
        const int o[5] = {b - 2 * BX, b - BX, b, b + BX, b + 2 * BX};
        R QM[NV];
        recon_window<R, NV>(s_prim, o, NB, weps, QM, Qz[m]);
        if (r < ez) V::store(s_z, (r + 1) * TX + lx, S::NZ, QM);
      }
    };
    auto z_fluxes = [&]() {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const int r = row + m * RPB - 1, f = r * TX + lx, b = bi0 + m * RPB * BX, kf = z0 + r;
        if (lx < ex && r >= 0 && r <= ez) {
          R QL[NV], F[NV];
          V::load(s_z, f, S::NZ, QL);
          const R pref = P::pf(Dl, kf);
          lmars<R, L>(C, QL, Qz[m], 2, pref, F);
          if constexpr (L::MOIST && MICRO) {
            // no condensate passes a wall (both z sides are)
            if (ph.sediment && kf != 0 && kf != nz) sediment_flux<R, L>(C, QL, Qz[m], pref, F);
          }
          if constexpr (VISC)
            viscous_flux<R, L>(C, P::ih(Dl, 2), s_prim, s_th, s_pi, b - BX, b, NB, F);
          V::store(s_z, f, S::NZ, F);
#pragma unroll
          for (int v = 0; v < NV; ++v) Qz[m][v] = F[v];
        }
      }
    };
    if constexpr (S::BOTH) {
      x_states();
#pragma unroll
      for (int m = 0; m < M; ++m) z_states(m);
      __syncthreads();
      x_fluxes();
      z_fluxes();
    } else {
      x_states();
      __syncthreads();
      x_fluxes();
      __syncthreads();
#pragma unroll
      for (int m = 0; m < M; ++m) {  // the face arrays of the two directions are separate
        x_divergence(m);
        z_states(m);
      }
      __syncthreads();
      z_fluxes();
    }
    if constexpr (S::PREFETCH && !RES) {
      if (stage != 0) cp_async_wait();  // this thread's own copies of Y^n
    }
    __syncthreads();
    const R dt = *s_dt;

    // ---- 3. z divergence, gravity source, stage combine, saturation adjustment, store
    R rate_max = R(0);
#pragma unroll
    for (int m = 0; m < M; ++m)
      if (owned(m)) {
        const int r = row + m * RPB - 1, k = z0 + r;
        if constexpr (S::BOTH) x_divergence(m);
        R F1[NV], yo[NV], mb = R(0), mt = R(0);
        V::load(s_z, (r + 1) * TX + lx, S::NZ, F1);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          acc[m][v] -= (F1[v] - Qz[m][v]) * P::ih(Dl, 2);
          if (v < L::IM0) mb += Qz[m][v], mt += F1[v];
        }
        const long long g = (long long)k * nx + (x0 + lx);
        finish_cell<R, L, MICRO>(
            a, Dl, ph, C, stage, dt, k, ys[m], acc[m], mb, mt,
            [&](int v) { return S::PREFETCH ? s_yn[(m * NV + v) * NT + tid] : Yn[v * ncell + g]; },
            yo);
#pragma unroll
        for (int v = 0; v < NV; ++v) Yo[v * ncell + g] = yo[v];
        if constexpr (RES) {
#pragma unroll
          for (int v = 0; v < NV; ++v) ys[m][v] = yo[v];
        }
        if (stage == 2)
          rate_max = fmax(rate_max, cell_rate_r<R, L>(C, yo, P::er(Dl, k), P::ih(Dl, 0), R(0),
                                                      P::ih(Dl, 2)));
      }
    if (stage == 2) {
      double bm;
      if constexpr (sizeof(R) == 4)
        bm = double(block_max_f(rate_max, reinterpret_cast<float *>(s_red + 1)));
      else
        bm = block_max(rate_max, s_red + 1);
      if (tid == 0)
        atomicMax(RES ? D.rate_next : D.rate, (unsigned long long)__double_as_longlong(bm));
    }
    __syncthreads();
  }
}

// The march along z (snap_march.cuh), for the tile shapes that ask for it.
template <class R, class L, class T>
struct MarchSmem;
template <class R, class L, class T, bool MICRO, bool RES>
__device__ __forceinline__ void march_tiles(const StageArgs &a, const int stage,
                                            unsigned char *smem);

// One stage over the CTA's tiles by the tile shape's method; st 0, 1, 2.
template <class R, class L, bool VISC, class T, bool MICRO>
__device__ __forceinline__ void run_stage(const StageArgs &a, int st, unsigned char *smem) {
  if constexpr (T::MARCH) {
    static_assert(!VISC, "the march is built for inviscid layouts");
    march_tiles<R, L, T, MICRO, false>(a, st, smem);
  } else if constexpr (L::D3) {
    R ys[Box<T, true>::CPT][L::NV];
    stage_tiles<R, L, VISC, T, MICRO>(a, st, smem, ys);
  } else {
    R ys[PlaneSmem<R, L, VISC, T>::M][L::NV];
    plane_tiles<R, L, VISC, T, MICRO>(a, st, smem, ys);
  }
}

// Cells per thread whose state the resident step keeps in registers.
template <class R, class L, bool VISC, class T>
constexpr int kept_cells() {
  if constexpr (T::MARCH)
    return 1;
  else if constexpr (L::D3)
    return Box<T, true>::CPT;
  else
    return PlaneSmem<R, L, VISC, T>::M;
}

template <class R, class L, bool VISC, class T>
constexpr size_t stage_smem() {
  if constexpr (T::MARCH)
    return MarchSmem<R, L, T>::total;
  else if constexpr (L::D3)
    return StageSmem<R, L, VISC, T>::total;
  else
    return PlaneSmem<R, L, VISC, T>::total;
}

// One Runge-Kutta stage over all tiles of all domains.
template <class R, class L, bool VISC, class T, bool MICRO>
__global__ void __launch_bounds__(T::NT, T::MINB) stage_kernel(const StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  run_stage<R, L, VISC, T, MICRO>(a, a.stage, smem);
}

// One whole step (three stages) in a single persistent cooperative launch: the CTAs walk the
// tile queue of every domain per stage and meet at a grid barrier between stages.
template <class R, class L, bool VISC, class T, bool MICRO>
__global__ void __launch_bounds__(T::NT, T::MINB) step_kernel(const StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
#pragma unroll 1
  for (int st = 0; st < 3; ++st) {
    run_stage<R, L, VISC, T, MICRO>(a, st, smem);
    if (st < 2) grid_barrier(a.gsync, gridDim.x, a.flags, a.spin_limit, a.absent_cta);
  }
}

// One whole step in a single cooperative launch with one tile per CTA (every tile of the
// launch co-resident): each CTA keeps its tile's state in registers through the three stages
// and, between stages, waits only for the tiles its ghost cells come from -- a flag per tile,
// set to 3 seq + s + 1 once the tile's stage-s output is in memory (seq counts the launches) --
// instead of a grid barrier or a new launch. Waits are bounded like the grid barrier's. The
// last CTA to finish moves each domain's next CFL rate into place and advances seq.
template <class R, class L, bool VISC, class T, bool MICRO, int MINB>
__global__ void __launch_bounds__(T::NT, MINB) resident_step_kernel(const StageArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned int s_seq;
  R ys[kept_cells<R, L, VISC, T>()][L::NV];
  const int tile = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) s_seq = ld_acquire_u32(&a.res->seq);
  __syncthreads();
  const unsigned int seq = s_seq;
  const int d0 = a.dep_begin[tile], nd = a.dep_begin[tile + 1] - d0;
#pragma unroll 1
  for (int st = 0; st < 3; ++st) {
    if (st > 0) {
      // the tiles this one's ghost cells come from have finished stage st - 1
      const unsigned int want = 3u * seq + unsigned(st);
      for (int i = tid; i < nd; i += blockDim.x) {
        const unsigned int *f = a.tile_flags + a.dep_list[d0 + i];
        const long long t0 = clock64();
        while (int(ld_acquire_u32(f) - want) < 0) {
          if (clock64() - t0 > a.spin_limit) {
            atomicOr(a.flags, (unsigned)kFlagTimeout);
            break;
          }
          __nanosleep(20);
        }
      }
      __syncthreads();
    }
    // either ends with a CTA barrier
    if constexpr (T::MARCH)
      march_tiles<R, L, T, MICRO, true>(a, st, smem);
    else if constexpr (L::D3)
      stage_tiles<R, L, VISC, T, MICRO, true>(a, st, smem, ys);
    else
      plane_tiles<R, L, VISC, T, MICRO, true>(a, st, smem, ys);
    if (st < 2 && tid == 0) {
      __threadfence();
      st_release_u32(a.tile_flags + tile, 3u * seq + unsigned(st) + 1u);
    }
  }
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(&a.res->done, 1u) == gridDim.x - 1) {
      __threadfence();
      for (int d = 0; d < a.ndom; ++d) {
        const DomDev &D = a.doms[d];
        *D.rate = atomicExch(D.rate_next, 0ull);
      }
      a.res->done = 0u;
      __threadfence();
      st_release_u32(&a.res->seq, seq + 1u);
    }
  }
}

// ------------------------------------------------------------------------------------------
// auxiliary kernels: CFL rate, budget, saturation adjustment over a domain
// ------------------------------------------------------------------------------------------
// The blocks take (level, chunk of blockDim.x cells of the level) items in turn, so the level
// of a cell comes from one division per item, not one per cell.
template <class R, class L>
__global__ void __launch_bounds__(256) rate_kernel(const StageArgs a, int dm, int buf) {
  __shared__ double red[32];
  const DomDev &D = a.doms[dm];
  const R *Y = reinterpret_cast<const R *>(D.buf[buf]);
  const long long plane = (long long)D.nx * D.ny;
  const long long chunks = (plane + blockDim.x - 1) / blockDim.x;
  const long long items = chunks * D.nz;
  double r = 0.0;
  for (long long it = blockIdx.x; it < items; it += gridDim.x) {
    const int k = int(it / chunks);
    const long long p = (it - k * chunks) * blockDim.x + threadIdx.x;
    if (p < plane) {
      const long long c = k * plane + p;
      R y[L::NV];
#pragma unroll
      for (int v = 0; v < L::NV; ++v) y[v] = Y[v * D.ncell + c];
      r = fmax(r, double(cell_rate_r<R, L>(cst<R>(a), y, Prof<R>::er(D, k), Prof<R>::ih(D, 0),
                                           Prof<R>::ih(D, 1), Prof<R>::ih(D, 2))));
    }
  }
  double bm = block_max(r, red);
  if (threadIdx.x == 0) atomicMax(D.rate, (unsigned long long)__double_as_longlong(bm));
}

// A caller-layout state (type S: energy as rho e) into the stored state of domain dm (type R,
// energy as rho e - e_ref of the level, the difference formed in FP64), with the CFL rate of
// the stored cells folded into the domain's rate slot: the state copy and the rate kernel in
// one pass. Items as in rate_kernel; VW consecutive cells of a level per thread, each field
// one aligned access (VW = 4 where every level starts on such a boundary, else 1).
template <class S, class R, class L, int VW>
__global__ void __launch_bounds__(256) load_rate_kernel(const S *src, const StageArgs a, int dm) {
  __shared__ double red[32];
  const DomDev &D = a.doms[dm];
  R *Y = reinterpret_cast<R *>(D.buf[0]);
  const long long plane = (long long)D.nx * D.ny, ncell = D.ncell;
  const long long span = (long long)blockDim.x * VW;
  const long long chunks = (plane + span - 1) / span;
  const long long items = chunks * D.nz;
  const CstT<R> &C = cst<R>(a);
  double r = 0.0;
  for (long long it = blockIdx.x; it < items; it += gridDim.x) {
    const int k = int(it / chunks);
    const long long p = (it - k * chunks) * span + (long long)threadIdx.x * VW;
    if (p < plane) {  // VW divides plane, so all VW cells lie in the level
      const long long c0 = k * plane + p;
      const double er = D.e_ref[k];
      R y[VW][L::NV];
#pragma unroll
      for (int v = 0; v < L::NV; ++v) {
        const Pack<S, VW> in = *reinterpret_cast<const Pack<S, VW> *>(src + v * ncell + c0);
        Pack<R, VW> out;
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          out.x[e] = v == L::IE ? R(double(in.x[e]) - er) : R(in.x[e]);
          y[e][v] = out.x[e];
        }
        *reinterpret_cast<Pack<R, VW> *>(Y + v * ncell + c0) = out;
      }
#pragma unroll
      for (int e = 0; e < VW; ++e)
        r = fmax(r, double(cell_rate_r<R, L>(C, y[e], Prof<R>::er(D, k), Prof<R>::ih(D, 0),
                                             Prof<R>::ih(D, 1), Prof<R>::ih(D, 2))));
    }
  }
  double bm = block_max(r, red);
  if (threadIdx.x == 0) atomicMax(D.rate, (unsigned long long)__double_as_longlong(bm));
}

// Per-block FP64 partial sums in a fixed order: nv field totals and sum(rho e + rho g z),
// all times the cell volume.
template <class R, class L>
__global__ void __launch_bounds__(256) budget_kernel(const StageArgs a, int dm, int buf,
                                                     double *partials) {
  constexpr int NO = L::NV + 1;
  __shared__ double red[NO][8];
  const DomDev &D = a.doms[dm];
  const R *Y = reinterpret_cast<const R *>(D.buf[buf]);
  const double vol = D.dx * (D.ny > 1 ? D.dy : 1.0) * D.dz;
  const long long plane = (long long)D.nx * D.ny;
  double s[NO];
#pragma unroll
  for (int o = 0; o < NO; ++o) s[o] = 0.0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < D.ncell;
       c += (long long)gridDim.x * blockDim.x) {
    const long long k = c / plane;
    const double z = (double(k) + 0.5) * D.dz;
    const double er = D.e_ref[k];
    double rho = 0.0;
#pragma unroll
    for (int v = 0; v < L::NV; ++v) {
      double y = double(Y[v * D.ncell + c]);
      if (v == L::IE) y += er;
      s[v] += y;
      if (v < L::IM0) rho += y;
    }
    s[L::NV] += (double(Y[(long long)L::IE * D.ncell + c]) + er) + rho * D.grav * z;
  }
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    double v = s[o];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[o][threadIdx.x >> 5] = v;
  }
  __syncthreads();
  if (threadIdx.x < NO) {
    double t = 0.0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) t += red[threadIdx.x][w];
    partials[(long long)blockIdx.x * NO + threadIdx.x] = t * vol;
  }
}

// Second pass of the budget: sums the per-block partials in block order (deterministic).
template <int Dummy = 0>
__global__ void budget_finish_kernel(const double *partials, int nblocks, int no, double *out) {
  for (int o = threadIdx.x; o < no; o += blockDim.x) {
    double t = 0.0;
    for (int b = 0; b < nblocks; ++b) t += partials[(long long)b * no + o];
    out[o] = t;
  }
}

template <class R, class L>
__global__ void __launch_bounds__(256) satadj_kernel(const StageArgs a, int dm, int buf) {
  const DomDev &D = a.doms[dm];
  R *Y = reinterpret_cast<R *>(D.buf[buf]);
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < D.ncell;
       c += (long long)gridDim.x * blockDim.x) {
    R y[L::NV];
#pragma unroll
    for (int v = 0; v < L::NV; ++v) y[v] = Y[v * D.ncell + c];
    const int k = int(c / ((long long)D.nx * D.ny));
    const int it = satadj_cell<R, L>(a.ph, cst<R>(a), y, Wide<R>::e_ref(D, k), Prof<R>::er(D, k),
                                     a.ph.satadj_max_iter);
    if (it < 0)
      atomicOr(a.flags, (unsigned)kFlagNoConv);
    else
      atomicMax(a.max_sweeps, it);
#pragma unroll
    for (int v = 0; v < L::NV; ++v) Y[v * D.ncell + c] = y[v];
  }
}

// ------------------------------------------------------------------------------------------
// host launchers of one configuration
// ------------------------------------------------------------------------------------------
template <class R, class L, bool VISC, class T, bool MICRO = false>
struct Variant {
  static constexpr size_t kSmem = stage_smem<R, L, VISC, T>();
  // the resident step as compiled for its most tiles per SM, and for one (the same but for FP64 with
  // one vapour)
  static constexpr auto kResident = &resident_step_kernel<R, L, VISC, T, MICRO, T::RESB>;
  static constexpr auto kOnePerSm = &resident_step_kernel<R, L, VISC, T, MICRO, T::MINB>;
  static cudaError_t prepare() {
    cudaError_t e = cudaFuncSetAttribute(stage_kernel<R, L, VISC, T, MICRO>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(kSmem));
    if (e != cudaSuccess) return e;
    for (const auto k : {kResident, kOnePerSm}) {
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
      if (e != cudaSuccess) return e;
    }
    return cudaFuncSetAttribute(step_kernel<R, L, VISC, T, MICRO>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
  }
  static int max_resident_tiles() {
    int dev = 0, nsm = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kResident, T::NT, kSmem) != cudaSuccess)
      return 0;
    return per * nsm;
  }
  static cudaError_t resident(const StageArgs &a, int grid, cudaStream_t s) {
    int dev = 0, nsm = 0;
    if (kResident != kOnePerSm) {
      cudaError_t e = cudaGetDevice(&dev);
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(T::NT);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, grid <= nsm ? kOnePerSm : kResident, a);
  }
  static cudaError_t stage(const StageArgs &a, int grid, cudaStream_t s) {
    stage_kernel<R, L, VISC, T, MICRO><<<grid, T::NT, kSmem, s>>>(a);
    return cudaGetLastError();
  }
  static int max_resident_blocks() {
    int dev = 0, nsm = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_kernel<R, L, VISC, T, MICRO>, T::NT,
                                                      kSmem) != cudaSuccess)
      return 0;
    return per * nsm;
  }
  static cudaError_t step(const StageArgs &a, int grid, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(T::NT);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, step_kernel<R, L, VISC, T, MICRO>, a);
  }
  static TileVariant get() {
    TileVariant v;
    v.tile[0] = T::TX;
    v.tile[1] = T::TY;
    v.tile[2] = T::TZ;
    v.levels = T::MARCH ? kMarchLevels : (L::D3 ? kFixedLevels : kPlaneLevels);
    v.fp64 = sizeof(R) == 8;
    v.threads = T::NT;
    v.smem_stage = kSmem;
    v.stage = &stage;
    v.step = &step;
    v.max_resident_blocks = &max_resident_blocks;
    v.prepare = &prepare;
    v.resident = &resident;
    v.max_resident_tiles = &max_resident_tiles;
    return v;
  }
};

template <class R, class L>
struct Family {
  static cudaError_t rate(const StageArgs &a, int dm, int buf, cudaStream_t s) {
    rate_kernel<R, L><<<304, 256, 0, s>>>(a, dm, buf);
    return cudaGetLastError();
  }
  template <class S>
  static cudaError_t load_typed(const void *src, const StageArgs &a, int dm, long long plane,
                                long long nz, cudaStream_t s) {
    const long long span = 256ll * 4, chunks = (plane + span - 1) / span;
    const long long items = chunks * nz;
    const int grid = int(items < 1216 ? items : 1216);
    if (plane % 4 == 0 && (uintptr_t)src % (4 * sizeof(S)) == 0)
      load_rate_kernel<S, R, L, 4><<<grid, 256, 0, s>>>((const S *)src, a, dm);
    else
      load_rate_kernel<S, R, L, 1><<<grid, 256, 0, s>>>((const S *)src, a, dm);
    return cudaGetLastError();
  }
  static cudaError_t load(const void *src, int src_f32, const StageArgs &a, int dm,
                          long long plane, long long nz, cudaStream_t s) {
    return src_f32 ? load_typed<float>(src, a, dm, plane, nz, s)
                   : load_typed<double>(src, a, dm, plane, nz, s);
  }
  static cudaError_t budget(const StageArgs &a, int dm, int buf, double *partials, int nblocks,
                            double *out, cudaStream_t s) {
    budget_kernel<R, L><<<nblocks, 256, 0, s>>>(a, dm, buf, partials);
    budget_finish_kernel<><<<1, 32, 0, s>>>(partials, nblocks, L::NV + 1, out);
    return cudaGetLastError();
  }
  static cudaError_t satadj(const StageArgs &a, int dm, int buf, cudaStream_t s) {
    satadj_kernel<R, L><<<608, 256, 0, s>>>(a, dm, buf);
    return cudaGetLastError();
  }
  // The tile shapes offered to the autotuner; the first is the default.
  template <bool VISC, class... Ts>
  static KernelSet set() {
    KernelSet k;
    k.nvariants = 0;
    TileVariant vs[] = {Variant<R, L, VISC, Ts>::get()...};
    for (const TileVariant &v : vs) k.var[k.nvariants++] = v;
    k.rate = &rate;
    k.load = &load;
    k.budget = &budget;
    k.satadj = &satadj;
    return k;
  }
  // kernels with the sedimentation fluxes and the Kessler scheme compiled in (inviscid)
  template <class... Ts>
  static KernelSet set_micro() {
    KernelSet k;
    k.nvariants = 0;
    TileVariant vs[] = {Variant<R, L, false, Ts, true>::get()...};
    for (const TileVariant &v : vs) k.var[k.nvariants++] = v;
    k.rate = &rate;
    k.load = &load;
    k.budget = &budget;
    k.satadj = &satadj;
    return k;
  }
};

}  // namespace snap
