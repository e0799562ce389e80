// One lane's share of a fused lattice update in which a warp works on rows of a strip of 64
// lattice columns, two adjacent ones per lane: shared by the warp sweep (lbm_sweep.cuh) and the
// tile kernel (lbm_tile.cuh).
//
// The 9-point stencils are separable: with s = c + (up + down)/4 and d = up - down of a
// column's three rows,
//   g_x = s_E - s_W,   g_y = d + (d_E + d_W)/4,   L = s_E + s_W + (up + down) - 5 c
// are the gradient and Laplacian sums of rk_rate (lbm_fused_tile.cuh), so a stage takes four
// shuffles for its two columns instead of nine shared-memory reads for one.  The two
// columns of a lane are the two lanes of the packed FP32 instructions: every operation of a
// node that is not an approximate reciprocal or root is half an instruction.
//
// With the energy equation the outer 5 columns on each side are halo (54 of 64 columns are
// outputs); without it one pair of columns (60 outputs).  Halo nodes are recomputed by the
// same instructions, so a node has the same bits whichever warp and column slot own it.
#pragma once

#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

namespace {

using V = float2;  // the values of a lane's two columns

__device__ __forceinline__ V vset(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ V vdup(float a) { return make_float2(a, a); }
__device__ __forceinline__ V operator+(V a, V b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ V operator*(V a, V b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ V vfma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
// a - b as (-1) b + a: rounds once, like the subtraction
__device__ __forceinline__ V operator-(V a, V b) { return __ffma2_rn(vdup(-1.0f), b, a); }
__device__ __forceinline__ float rcp_approx(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ V vrcp(V a) { return vset(rcp_approx(a.x), rcp_approx(a.y)); }
// a copy through the packed adder: one instruction for the pair instead of two moves
__device__ __forceinline__ V vcopy(V a) {
  return __fadd2_rn(a, make_float2(0.0f, 0.0f));
}
__device__ __forceinline__ V vsqrt(V a) { return vset(sqrtf(a.x), sqrtf(a.y)); }
__device__ __forceinline__ V vrsqrt(V a) { return vset(rsqrtf(a.x), rsqrtf(a.y)); }

// A constant operand.  The two-lane instructions take it as a register pair that holds it
// twice (PACK), which pays for constants used several times a step; one used once costs more
// instructions to put into a pair than two scalar operations with the constant as an
// immediate or from the constant bank (4096 x 512: 48.6 us per update with this split, 50.6
// with every constant in a pair; 16384 x 2048: 575 and 617 us).
template <bool PACK>
struct KC {
  float v;
};
using KL = KC<true>;   // literal
using KP = KC<true>;   // parameter used several times a step
using K1 = KC<false>;  // parameter or literal used once a step
template <bool PK>
__device__ __forceinline__ V operator*(KC<PK> c, V a) {
  return PK ? __fmul2_rn(vdup(c.v), a) : vset(c.v * a.x, c.v * a.y);
}
template <bool PK>
__device__ __forceinline__ V operator+(KC<PK> c, V a) {
  return PK ? __fadd2_rn(vdup(c.v), a) : vset(c.v + a.x, c.v + a.y);
}
template <bool PK>
__device__ __forceinline__ V vfma(KC<PK> c, V a, V b) {
  return PK ? __ffma2_rn(vdup(c.v), a, b) : vset(fmaf(c.v, a.x, b.x), fmaf(c.v, a.y, b.y));
}
// a c + k with a constant addend
template <bool PK>
__device__ __forceinline__ V vfma(V a, V b, KC<PK> c) {
  return PK ? __ffma2_rn(a, b, vdup(c.v)) : vset(fmaf(a.x, b.x, c.v), fmaf(a.y, b.y, c.v));
}
template <bool PA, bool PB>
__device__ __forceinline__ V vfma(KC<PA> c, V a, KC<PB> d) {
  return PA && PB ? __ffma2_rn(vdup(c.v), a, vdup(d.v))
                  : vset(fmaf(c.v, a.x, d.v), fmaf(c.v, a.y, d.v));
}
// c - a
template <bool PK>
__device__ __forceinline__ V operator-(KC<PK> c, V a) {
  return PK ? vdup(c.v) - a : vset(c.v - a.x, c.v - a.y);
}
__device__ __forceinline__ KL kl(float v) { return KL{v}; }
__device__ __forceinline__ KP kp(float v) { return KP{v}; }
__device__ __forceinline__ K1 k1(float v) { return K1{v}; }

constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ int modi(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// columns of halo on each side of a warp's outputs, and its output columns
__host__ __device__ constexpr int sweep_halo(bool th) { return th ? 5 : 2; }
__host__ __device__ constexpr int sweep_width(bool th) { return 64 - 2 * sweep_halo(th); }
// rows of halo below and above a chunk
__host__ __device__ constexpr int sweep_rows(bool th) { return th ? 5 : 1; }
// first even column of strip k (outputs [c + halo, c + halo + width), clipped to the
// lattice)
__host__ __device__ constexpr int sweep_c0(int k, bool th) {
  return k * sweep_width(th) - (th ? 6 : 2);
}
__host__ __device__ constexpr int sweep_strips(int nx, bool th) {
  return (nx + (th ? 1 : 0) + sweep_width(th) - 1) / sweep_width(th);
}

inline SweepConsts sweep_consts(const DevParams &p) {
  SweepConsts k;
  k.rho_ref = p.rho_ref;
  k.b = p.eos_b;
  k.inv_Tc = p.inv_Tc;
  k.xr = p.xr;
  k.sr = p.sr;
  k.nkappa = -p.kappa;
  k.kappa1r = p.kappa1 + p.rphi_r;
  k.ps_g = p.ps_g;
  k.ps_RT = p.ps_RT;
  k.ps_R = p.ps_R;
  k.ps_phi = p.ps_phi;
  k.ps_B = p.ps_B;
  k.ps_3 = p.ps_3;
  k.psi_r2 = p.psi_r2;
  // the denominator psi + psi_r stays positive where both vanish (the quotient is 0 there)
  k.psi_den = std::max(p.psi_r, 1e-30f);
  k.akap1_cv3 = p.akap1_cv3;
  k.nkappa_r = -p.kappa_r;
  k.RTc_cv3 = p.RTc_cv3;
  k.lam23_cv = p.lam23_cv;
  k.G3 = p.G3;
  k.G3r = p.G3r;
  k.nk10 = -p.k1[0];
  k.k11 = p.k1[1];
  k.k12 = p.k1[2];
  k.k13 = p.k1[3];
  k.k14 = p.k1[4];
  k.k20 = p.k2[0];
  k.k21 = p.k2[1];
  k.k22 = p.k2[2];
  k.k23 = p.k2[3];
  k.k24 = p.k2[4];
  k.kq0 = p.kq[0];
  k.kq1 = p.kq[1];
  k.kq2 = p.kq[2];
  k.kn0 = p.kn[0];
  k.kn1 = p.kn[1];
  k.kn2 = p.kn[2];
  k.kn3 = p.kn[3];
  return k;
}

// Loads of one population and of an aligned column pair, converted as the storage's load
// does.  Plain (coherent) loads: the kernel may start while the previous update still runs,
// and a read-only load could be moved above its wait for that update.
template <class ST>
__device__ __forceinline__ float pop(const typename ST::T *p, int i);
template <>
__device__ __forceinline__ float pop<StoreF32>(const float *p, int) { return *p; }
template <>
__device__ __forceinline__ float pop<StoreBF16>(const __nv_bfloat16 *p, int i) {
  return wlat(i) * __bfloat162float(*p);
}
template <>
__device__ __forceinline__ float pop<StoreF16>(const __half *p, int i) {
  return wlat(i) * __half2float(*p);
}
template <class ST>
__device__ __forceinline__ V pop2(const typename ST::T *p, int i);
template <>
__device__ __forceinline__ V pop2<StoreF32>(const float *p, int) {
  return *reinterpret_cast<const float2 *>(p);
}
template <>
__device__ __forceinline__ V pop2<StoreBF16>(const __nv_bfloat16 *p, int i) {
  const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
  return vset(wlat(i) * v.x, wlat(i) * v.y);
}
template <>
__device__ __forceinline__ V pop2<StoreF16>(const __half *p, int i) {
  const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(p));
  return vset(wlat(i) * v.x, wlat(i) * v.y);
}

// One lane of a warp that works on rows of a strip of 64 columns: its geometry, boundary
// cases, loads and the arithmetic of the update, for the lane's two columns at once.
template <bool YW, bool XO, bool TH, bool MP, class ST>
struct Lane {
  using T = typename ST::T;
  static constexpr int HR = sweep_rows(TH);  // halo rows
  static constexpr int HC = sweep_halo(TH);  // halo columns
  static constexpr unsigned E = sizeof(T);

  const DevParams &p;
  const SweepConsts &k;
  const T *gs;
  T *gout;
  const float *Tin;
  float *Tout;
  const StepScalars &sc;
  // Geometry of the lane: its first column c0 (even), the lattice column x0 it loads from
  // (c0 wrapped into a periodic lattice, clamped beyond an open end, where the loaded
  // values are replaced or never used), and element offsets from x0 to the second column
  // (o1), the west source of the first (oW) and the east source of the second (oE).
  int c0, x0, o1, oW, oE;
  bool vec;            // the column pair is one aligned pair of elements
  bool e_in, e_out, ends;  // the warp holds the inlet (outlet) column or its ghost; either
  bool has_g, tau_const;
  float in_u;          // velocity inlet: U / (1 - U)
  bool outp;           // the lane stores its pair's populations
  bool out_x, out_y;   // the first (second) column is column nx - 1
  bool oddx;           // the second column of the pair lies beyond the lattice
  bool out0, out1;     // output columns

  struct Own {  // values of a node that its RK4 stages share
    V nux, nuy, cl, Tb, nE1, nE2;
  };

  V g[9], Tn;              // populations and temperature of a row as loaded
  unsigned st;
  float drho_min, drho_max, dT_min;
  V chk;                   // not finite once a stored value is not

  __device__ __forceinline__ Lane(const DevParams &p_, const SweepConsts &k_, const T *gs_, T *gout_,
                                  const float *Tin_, float *Tout_, const StepScalars &sc_, int C0)
      : p(p_), k(k_), gs(gs_), gout(gout_), Tin(Tin_), Tout(Tout_), sc(sc_) {
    const int lane = (int)(threadIdx.x & 31);
    c0 = C0 + 2 * lane;
    o1 = 1;
    oW = -1;
    oE = 2;
    if (XO) {
      x0 = min(max(c0, 0), (p.nx - 1) & ~1);
      vec = true;
    } else {
      x0 = modi(c0, p.nx);
      o1 = modi(c0 + 1, p.nx) - x0;
      oW = modi(c0 - 1, p.nx) - x0;
      oE = modi(c0 + 2, p.nx) - x0;
      vec = (p.nx & 1) == 0;
    }
    in_u = XO ? sc.u_in / (1.0f - sc.u_in) : 0.0f;
    has_g = p.has_g;
    tau_const = p.tau_const;
    e_in = XO && C0 <= 0;
    e_out = XO && C0 + 63 >= p.nx - 1;
    ends = e_in || e_out;
    out_x = XO && c0 == p.nx - 1;
    out_y = XO && c0 + 1 == p.nx - 1;
    const bool in0 = c0 >= 0 && c0 < p.nx, in1 = c0 + 1 >= 0 && c0 + 1 < p.nx;
    outp = lane >= HC / 2 && lane < 32 - HC / 2 && in0;
    oddx = !in1;
    out0 = 2 * lane >= HC && 2 * lane < 64 - HC && in0;
    out1 = 2 * lane + 1 >= HC && 2 * lane + 1 < 64 - HC && in1;
    const V z = vdup(0.0f);
#pragma unroll
    for (int i = 0; i < 9; i++) g[i] = z;
    Tn = chk = z;
    st = 0u;
    drho_min = drho_max = dT_min = 0.0f;
  }

  // ---- neighbour columns and open ends ----
  // West neighbour of the first column and east neighbour of the second, from the lanes
  // beside.  Ghost columns beyond an open end (fix: some warps of the strip only): the outlet
  // ghost, column nx, copies column nx - 1, so that column is its own east neighbour; the
  // inlet ghost, column -1, is either a column of its own values or (copy_in) copies column 0.
  __device__ __forceinline__ void neighbours(V &a, bool copy_in, float &w, float &e) const {
    if (XO && ends && out_x) a.y = a.x;
    w = __shfl_up_sync(kAll, a.y, 1);
    e = __shfl_down_sync(kAll, a.x, 1);
    if (XO && ends) {
      if (out_y) e = a.y;
      if (copy_in && c0 == 0) w = a.x;
    }
  }
  // Separable sums of a 9-point stencil (see the file comment): g_x, g_y and, for the
  // Laplacian, s_E + s_W and up + down.  (The neighbours inside the pair are the lane's own
  // registers: scalar operations take them as they are, a packed one would first copy them
  // into a register pair.)
  struct Sten {
    V gx, gy, es, a;
  };
  __device__ __forceinline__ Sten stencil(V dn, V c, V up, bool copy_in) const {
    Sten r;
    r.a = up + dn;
    const KL q = kl(0.25f);
    V s = vfma(q, r.a, c), d = up - dn;
    float w, e, dw, de;
    neighbours2(s, d, copy_in, w, e, dw, de);
    r.gx = vset(s.y - w, e - s.x);
    r.es = vset(s.y + w, e + s.x);
    r.gy = vfma(q, vset(d.y + dw, de + d.x), d);
    return r;
  }
  __device__ __forceinline__ void neighbours2(V &s, V &d, bool copy_in, float &w, float &e,
                                              float &dw, float &de) const {
    if (XO && ends) {
      neighbours(s, copy_in, w, e);
      neighbours(d, copy_in, dw, de);
    } else {
      w = __shfl_up_sync(kAll, s.y, 1);
      e = __shfl_down_sync(kAll, s.x, 1);
      dw = __shfl_up_sync(kAll, d.y, 1);
      de = __shfl_down_sync(kAll, d.x, 1);
    }
  }

  __device__ __forceinline__ bool ghost(int j) const {
    return XO && (c0 + j < 0 || c0 + j >= p.nx);
  }
  // the inlet ghost, column -1, is the second column of the lane with c0 = -2
  __device__ __forceinline__ V inlet_set(V a, float v) const {
    if (c0 == -2) a.y = v;
    return a;
  }
  // Zou-He on the boundary columns of row r (see pull_fix): every lane computes the rule on
  // its own column, the boundary column's lane keeps the result
  __device__ __forceinline__ void inlet_fix(int r) {
    const float known = g[0].x + g[2].x + g[4].x + 2.0f * (g[3].x + g[6].x + g[7].x);
    // momentum rho U of the end: the pressure inlet gives rho, U = 1 - (known + rho_ref) / rho;
    // the velocity inlet gives U, rho = (known + rho_ref) / (1 - U) (in_u = U / (1 - U))
    const float m = p.p_inlet ? sc.rho_in - p.rho_ref - known : (known + p.rho_ref) * in_u;
    const float g1 = fmaf(2.0f / 3.0f, m, g[3].x);
    const float d24 = 0.5f * (g[2].x - g[4].x), m6 = m * (1.0f / 6.0f);
    const float g5 = (g[7].x - d24) + m6, g8 = (g[6].x + d24) + m6;
    const bool me = c0 == 0;
    if (me) g[1].x = g1;
    if (me && !(YW && r == 0)) g[5].x = g5;  // the link from below is a fluid one
    if (me && !(YW && r == p.ny - 1)) g[8].x = g8;
  }
  __device__ __forceinline__ void outlet_rule(const float (&f)[9], float &f3, float &f6,
                                              float &f7) const {
    // momentum rho U of the end
    const float m = f[0] + f[2] + f[4] + 2.0f * (f[1] + f[5] + f[8]) + (p.rho_ref - p.rho_out);
    const float d24 = 0.5f * (f[2] - f[4]), m6 = m * (1.0f / 6.0f);
    f3 = fmaf(-2.0f / 3.0f, m, f[1]);
    f7 = (f[5] + d24) - m6;
    f6 = (f[8] - d24) - m6;
  }
  __device__ __forceinline__ void outlet_fix(int r) {
    const bool lo = YW && r == 0, hi = YW && r == p.ny - 1, odd = (p.nx & 1) != 0;
    float f[9], f3, f6, f7;
#pragma unroll
    for (int i = 0; i < 9; i++) f[i] = odd ? g[i].x : g[i].y;
    outlet_rule(f, f3, f6, f7);
    const bool mx = out_x, my = out_y;
    if (mx) g[3].x = f3;
    if (my) g[3].y = f3;
    if (mx && !lo) g[6].x = f6;
    if (my && !lo) g[6].y = f6;
    if (mx && !hi) g[7].x = f7;
    if (my && !hi) g[7].y = f7;
  }

  // ---- walls ----
  // a stage field on solid row q: the wall temperature; the top ghost of an adiabatic
  // column copies row ny - 1 (`below`, the row swept before)
  __device__ __forceinline__ V wall_T(int q, V below) const {
    float w[2];
#pragma unroll
    for (int j = 0; j < 2; j++) {
      const int x = XO ? c0 + j : (j ? x0 + o1 : x0);
      w[j] = q < 0 ? wall_T_dev(p, x) : wall_T_top_dev(p, x);
      if (!XO && q >= 0 && p.adiabatic && wall_adiabatic(p, x, true)) w[j] = j ? below.y : below.x;
    }
    return vset(w[0], w[1]);
  }
  // the bottom ghost of an adiabatic column copies row 0: once row 0 has its value v, it goes
  // into the ghost row's slot
  __device__ __forceinline__ void mirror_bottom(V &slot, V v) const {
    if (!XO && p.adiabatic) {
      if (wall_adiabatic(p, x0, false)) slot.x = v.x;
      if (wall_adiabatic(p, x0 + o1, false)) slot.y = v.y;
    }
  }
  // ---- loads ----
  // element at byte offset b (32-bit) from a uniform base
  template <class X>
  static __device__ __forceinline__ X *at(X *base, unsigned b) {
    return const_cast<X *>(
        reinterpret_cast<const X *>(reinterpret_cast<const char *>(base) + b));
  }
  // issue the loads of row r; near: it may be a wall row or next to one
  __device__ __forceinline__ void load_row(bool near, int r) {
    if (YW && near && (unsigned)r >= (unsigned)p.ny) return;
    const int ry = YW ? r : modi(r, p.ny);
    const unsigned R = (unsigned)(ry * p.pitch + x0);  // element offset in a plane
    if (YW && near && (ry == 0 || ry == p.ny - 1)) {
      // next to a wall: links from the solid row come from the node's own opposite
      // population (half-way bounce-back; the weights of the two are the same)
#pragma unroll
      for (int i = 0; i < 9; i++) {
        const bool back = (ey(i) == 1 && ry == 0) || (ey(i) == -1 && ry == p.ny - 1);
        const int e = back ? 0 : ex(i);
        const T *b = gs + (back ? opp(i) * p.plane : i * p.plane - ey(i) * p.pitch) + R;
        const int a = e == 0 ? 0 : (e == 1 ? oW : o1);
        const int c = e == 0 ? o1 : (e == 1 ? 0 : oE);
        g[i] = vset(pop<ST>(b + a, i), pop<ST>(b + c, i));
      }
    } else {
      // rows below and above: offsets of their own where the rows wrap
      const unsigned Rm = YW ? R - p.pitch : (unsigned)(modi(ry - 1, p.ny) * p.pitch + x0);
      const unsigned Rp = YW ? R + p.pitch : (unsigned)(modi(ry + 1, p.ny) * p.pitch + x0);
#pragma unroll
      for (int i = 0; i < 9; i++) {
        const T *b = gs + i * p.plane;
        const unsigned o = (ey(i) == 0 ? R : (ey(i) == 1 ? Rm : Rp)) * E;
        if (XO) {
          // (planes 1 .. 8: a neighbour element is in bounds at the ends of the array too)
          if (ex(i) == 0) {
            g[i] = pop2<ST>(at(b, o), i);
          } else {
            g[i] = vset(pop<ST>(at(b, o) - ex(i), i), pop<ST>(at(b, o) - ex(i) + 1, i));
          }
        } else if (ex(i) == 0) {
          g[i] = vec ? pop2<ST>(at(b, o), i)
                     : vset(pop<ST>(at(b, o), i), pop<ST>(at(b, o) + o1, i));
        } else {
          g[i] = vset(pop<ST>(at(b, o) + (ex(i) == 1 ? oW : o1), i),
                      pop<ST>(at(b, o) + (ex(i) == 1 ? 0 : oE), i));
        }
      }
    }
    const float *t = at(Tin, 4u * R);
    Tn = vec ? *reinterpret_cast<const float2 *>(t) : vset(t[0], t[o1]);
  }

  // ---- the update of a row ----
  // the ends' populations and ghost temperature of row r as loaded
  __device__ __forceinline__ void open_ends(int r) {
    if (e_in) inlet_fix(r);
    if (e_out) outlet_fix(r);
    if (e_in) Tn = inlet_set(Tn, p.T_inlet_dev);
  }
  // the moments n = M g (Eq. 6) from sums and differences of opposite directions:
  // drho, -n1, n2, jx, n4, jy, n6, n7, n8
  __device__ __forceinline__ void moments(V (&n)[9]) const {
    const V s13 = g[1] + g[3], s24 = g[2] + g[4], s57 = g[5] + g[7], s68 = g[6] + g[8];
    const V d13 = g[1] - g[3], d24 = g[2] - g[4], d57 = g[5] - g[7], d68 = g[6] - g[8];
    const V sa = s13 + s24, sd = s57 + s68, f0 = g[0];
    const V dx = d57 - d68, dy = d57 + d68;
    n[0] = (f0 + sa) + sd;
    n[1] = vfma(kl(-2.0f), sd, vfma(kl(4.0f), f0, sa));
    n[2] = vfma(kl(-2.0f), sa, vfma(kl(4.0f), f0, sd));
    n[3] = d13 + dx;
    n[4] = vfma(kl(-2.0f), d13, dx);
    n[5] = d24 + dy;
    n[6] = vfma(kl(-2.0f), d24, dy);
    n[7] = s13 - s24;
    n[8] = s57 - s68;
  }
  // psi - psi_r (see pseudopotential_dev) and the energy coefficients E1 / (3 div u) and
  // E2 / (3 div u) of density and temperature deviations; neg: the argument of Eq. 10's root
  // is negative (psi = 0)
  __device__ __forceinline__ void state(V drho, V T_r, V &psi_r, V &cfx, V &cfz, bool &neg0,
                                        bool &neg1) const {
    if (!MP && !TH) return;
    const V rho = kp(k.rho_ref) + drho;
    const V br = k1(k.b) * rho;
    const V inv1 = vrcp(kl(1.0f) - br);
    const V invD = vrcp(vfma(br, kl(2.0f) - br, kl(1.0f)));
    if (TH) {
      cfz = (k1(k.akap1_cv3) * rho) * invD;
      cfx = vfma(k1(k.nkappa_r), cfz, k1(k.RTc_cv3) * inv1);
    }
    if (MP) {
      const V s = vsqrt(vfma(kp(k.inv_Tc), T_r, kp(k.xr)));
      const V ds = (kp(k.inv_Tc) * T_r) * vrcp(k1(k.sr) + s);
      const V rr = vfma(k1(k.nkappa), s, k1(k.kappa1r));  // r(T) + r(T_ref)
      const V gg = vfma(k1(k.ps_g), rho, kp(k.rho_ref));
      const V tR = inv1 * vfma(k1(k.ps_RT) * T_r, rho, k1(k.ps_R) * drho);
      const V tA = invD * vfma((k1(k.ps_phi) * ds) * rr, rho * rho, (k1(k.ps_B) * drho) * gg);
      const V dpsi2 = vfma(k1(k.ps_3), drho, tR - tA);
      const V psi2 = k1(k.psi_r2) + dpsi2;
      const V root = vsqrt(vset(fmaxf(psi2.x, 0.0f), fmaxf(psi2.y, 0.0f)));
      psi_r = dpsi2 * vrcp(k1(k.psi_den) + root);
      neg0 = !(psi2.x >= 0.0f);
      neg1 = !(psi2.y >= 0.0f);
      psi_r.x = neg0 ? -p.psi_r : psi_r.x;
      psi_r.y = neg1 ? -p.psi_r : psi_r.y;
    }
  }
  // running checks of a row's density and temperature deviations
  __device__ __forceinline__ void track(V dr, V dt, bool neg) {
    if (MP) st |= neg ? ST_PSI_NEG : 0u;
    drho_min = fminf(drho_min, fminf(dr.x, dr.y));
    drho_max = fmaxf(drho_max, fmaxf(dr.x, dr.y));
    dT_min = fminf(dT_min, fminf(dt.x, dt.y));
  }
  // forces of Eqs. 9, 14, 15 on row q from psi of rows q - 1 .. q + 1; wall: the row has a wall
  // neighbour; T_q: its temperature
  __device__ __forceinline__ void forces(int q, bool wall, V dn, V c, V up, V T_q, V drho, V &Fx,
                                         V &Fy, V &fm2) const {
    Fx = Fy = fm2 = vdup(0.0f);
    if (MP) {
      const Sten t = stencil(dn, c, up, true);
      const V gpsi = vfma(k1(k.G3), c, k1(k.G3r));  // -G psi / 3
      Fx = gpsi * t.gx;
      Fy = gpsi * t.gy;
      V qy = t.gy;
      if (wall) {
        // wall neighbours (psi of a solid row is 0 in the stencil): Eq. 14, see
        // interaction_force; Sy = 3 sum_solid w e_y
        const float Sy = (q == p.ny - 1 ? 1.5f : 0.0f) - (q == 0 ? 1.5f : 0.0f);
        float wc[2];
#pragma unroll
        for (int i = 0; i < 2; i++) {
          const float Tq = i ? T_q.y : T_q.x, pc = i ? c.y : c.x;
          unsigned unused = 0u;
          wc[i] = p.rho_w > 0.0f
                      ? p.G * p.psi_r - p.Gw * pseudopotential(p, p.rho_w, p.T_ref + Tq, unused)
                      : p.wall_r - p.Gw * pc;
        }
        const V ws = kl(1.0f / 3.0f) * (vdup(p.psi_r) + c) * vset(wc[0], wc[1]);
        Fy = vfma(ws, vdup(Sy), Fy);
        qy = vfma(vdup(-p.psi_r), vdup(Sy), qy);
      }
      fm2 = vfma(t.gx, t.gx, qy * qy);
    }
    if (has_g) {
      const V rv = vdup(p.drho_ref_g) + drho;  // rho - rho_v of Eq. 15
      Fx = Fx + rv * vdup(p.gx) * vdup(sc.gcos);
      Fy = Fy + rv * vdup(p.gy) * vdup(sc.gcos);
    }
  }
  // moment-space collision (see collide) of row q and the store of its populations
  __device__ __forceinline__ void collide_store(int q, const V (&n)[9], V rho, V jx, V jy, V u_x,
                                                V u_y, V Fx, V Fy, V fm2) {
    // moment-space collision (see collide): a_k = (m*_k - rho_ref c_k) / D_k
    const V uxF = u_x * Fx, uyF = u_y * Fy, uxj = jx * u_x, uyj = jy * u_y;
    const V uF = uxF + uyF, uu = uxj + uyj;
    const V dF = uxF - uyF, dj = uxj - uyj, xF = vfma(u_x, Fy, u_y * Fx), xj = jx * u_y;
    V a7, a8;
    if (tau_const) {
      a7 = vfma(k1(k.kn2), dF, vfma(kp(k.kn1), dj, kp(k.kn0) * n[7]));
      a8 = vfma(k1(k.kn3), xF, vfma(kp(k.kn1), xj, kp(k.kn0) * n[8]));
    } else {
      const float fx = fminf(fmaxf((rho.x - p.rho_g) * p.inv_drho, 0.0f), 1.0f);
      const float fy = fminf(fmaxf((rho.y - p.rho_g) * p.inv_drho, 0.0f), 1.0f);
      // c = 0.25 s_nu of Eq. 5
      const V c = kl(0.25f) * vrcp(vset(p.tau_g + fx * p.dtau, p.tau_g + fy * p.dtau));
      const V ca = kl(0.25f) - c;
      a7 = vfma(kl(0.5f) - c, dF, vfma(c, dj, ca * n[7]));
      a8 = vfma(vfma(kl(-0.5f), c, kl(0.25f)), xF, vfma(c, xj, ca * n[8]));
    }
    const V drho = n[0];
    const V a0 = k1(1.0f / 9.0f) * drho;
    const V a1 = vfma(k1(k.k14), fm2, vfma(k1(k.k13), uF, vfma(k1(k.k12), uu,
                          vfma(k1(k.k11), drho, k1(k.nk10) * n[1]))));
    const V a2 = vfma(k1(k.k24), fm2, vfma(k1(k.k23), uF, vfma(k1(k.k22), uu,
                          vfma(k1(k.k21), drho, k1(k.k20) * n[2]))));
    const V a3 = k1(1.0f / 6.0f) * (n[3] + Fx), a5 = k1(1.0f / 6.0f) * (n[5] + Fy);
    const V a4 = vfma(kp(k.kq2), Fx, vfma(kp(k.kq1), jx, kp(k.kq0) * n[4]));
    const V a6 = vfma(kp(k.kq2), Fy, vfma(kp(k.kq1), jy, kp(k.kq0) * n[6]));
    const KL m2 = kl(-2.0f);
    const V b_ax = vfma(m2, a2, a0 - a1), b_dg = vfma(kl(2.0f), a1, a0) + a2;
    const V px = vfma(m2, a4, a3), py = vfma(m2, a6, a5);
    const V tx = a3 + a4, ty = a5 + a6;
    const V qs = tx + ty, qd = ty - tx;
    const V axp = b_ax + a7, axm = b_ax - a7, dgp = b_dg + a8, dgm = b_dg - a8;
    V o[9];
    o[0] = vfma(kl(4.0f), a2 - a1, a0);
    o[1] = axp + px;
    o[2] = axm + py;
    o[3] = axp - px;
    o[4] = axm - py;
    o[5] = dgp + qs;
    o[6] = dgm + qd;
    o[7] = dgp - qs;
    o[8] = dgm - qd;
    V ck = u_x * u_y;  // not finite when either is not
    if (XO ? e_out : oddx) {
      // odd nx: the padding column stays zero
      if (oddx) {
        ck.y = 0.0f;
#pragma unroll
        for (int i = 0; i < 9; i++) o[i].y = 0.0f;
      }
    }
    // whole pairs: with the energy equation the pairs at the ends of the output columns
    // hold one halo column each, whose populations are complete here too; the
    // neighbouring warp stores the same bits
    if (outp) {
      chk = chk + ck;
      const unsigned so = (unsigned)((YW ? q : modi(q, p.ny)) * p.pitch + c0) * E;
#pragma unroll
      for (int i = 0; i < 9; i++) ST::store2(at(gout + i * p.plane, so), o[i].x, o[i].y, i);
    }
  }
  // the values of row q's nodes that the RK4 stages share, from the velocity of rows q - 1,
  // q (c) and q + 1
  __device__ __forceinline__ Own own_values(V uxd, V uxc, V uxu, V uyd, V uyc, V uyu, V cl, V Tb,
                                            V cfx, V cfz) const {
    const KL q4 = kl(0.25f);
    const K1 n3 = k1(-1.0f / 3.0f);
    V sx = vfma(q4, uxu + uxd, uxc), dy = uyu - uyd;
    float w, e, dw, de;
    neighbours2(sx, dy, p.p_inlet != 0, w, e, dw, de);
    const V nd =
        kl(-1.0f) * (vset(sx.y - w, e - sx.x) + vfma(q4, vset(dy.y + dw, de + dy.x), dy));
    Own o{n3 * uxc, n3 * uyc, cl, Tb, cfx * nd, cfz * nd};
    // the inlet ghost keeps T_inlet through the stages: no rate there
    if (XO && ends && c0 == -2) o.nux.y = o.nuy.y = o.cl.y = o.nE1.y = o.nE2.y = 0.0f;
    return o;
  }
  // K(T) of Eq. 16 (see rk_rate): -us.g + cl L - E1 x - E2 s
  __device__ __forceinline__ V rate(V dn, V c, V up, const Own &o) const {
    const Sten t = stencil(dn, c, up, false);
    const V lap = t.es + vfma(kl(-5.0f), c, t.a);
    const V x = vfma(kp(k.inv_Tc), c, kp(k.xr));  // T/Tc > 0 on fluid nodes
    const V s = x * vrsqrt(x);
    return vfma(o.nE2, s, vfma(o.nE1, x, vfma(o.cl, lap, vfma(o.nux, t.gx, o.nuy * t.gy))));
  }
  // the new temperature of row q
  __device__ __forceinline__ void store_T(int q, V Tnew) {
    const unsigned so = 4u * (unsigned)((YW ? q : modi(q, p.ny)) * p.pitch + c0);
    float *d = at(Tout, so);
    if (out0 && out1) {
      chk = chk + Tnew;
      dT_min = fminf(dT_min, fminf(Tnew.x, Tnew.y));
      *reinterpret_cast<float2 *>(d) = Tnew;
    } else if (out0 || out1) {
      const float v = out0 ? Tnew.x : Tnew.y;
      chk.x += v;
      dT_min = fminf(dT_min, v);
      if (out0) d[0] = v;
      if (out1) at(Tout, so + 4u)[0] = v;
    }
  }
  // the status bits of the running checks
  __device__ __forceinline__ void finish(unsigned *status) {
    if (!isfinite(chk.x + chk.y)) st |= ST_NAN;
    if (!(p.rho_ref + drho_min > 0.0f)) st |= ST_RHO_NONPOS;
    if (!(p.eos_b * (p.rho_ref + drho_max) < 1.0f)) st |= ST_EOS_POLE;
    if (!(p.T_ref + dT_min > 0.0f)) st |= ST_T_NONPOS;
    set_status(status, st);
  }
};

}  // namespace

}  // namespace lbm
