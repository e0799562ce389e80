// Fused lattice update on tiles of one row per warp.
//
// A CTA owns a strip of 64 lattice columns (two adjacent ones per lane) and a few rows; each
// warp holds one row of the tile or of its halo (5 rows on each side with the energy
// equation, 1 without) in its registers, from the loads to the stores.  The stages of the
// update are phases between barriers: in each, a warp reads the values of the rows below and
// above from shared memory, takes its neighbour columns by shuffles and publishes its own
// result:
//   0  pull-streaming with boundary rules (Eq. 12), moments, density, pseudopotential
//      (Eqs. 10-13)                                                        -> psi, T
//   1  forces (Eqs. 9, 14, 15), velocity (Eq. 13), MRT collision (Eqs. 6-8),
//      store of the populations                                            -> u
//   2  div u, h1 (Eqs. 16, 18)   3  h2   4  h3                             -> T2, T3, T4
//   5  h4 and Eq. 17, store of the temperature
// A phase has a row of work for every warp, so an update of a small lattice takes six short
// phases instead of the row-after-row pipeline of a sweep.  The lane's arithmetic is in
// lbm_lane.cuh, so a node has the same bits here and in the warp sweep.
#pragma once

#include "lbm_lane.cuh"

namespace lbm {

namespace {

// MAXW: most warps of a CTA
template <int MAXW>
struct TileSmem {
  float2 a[MAXW][32];  // psi, then T2, then T4
  float2 t[MAXW][32];  // T
  float2 b[MAXW][32];  // u_x, then T3
  float2 c[MAXW][32];  // u_y
};

template <bool YW, bool XO, bool TH, bool MP, class ST, int MAXW>
struct Tile : Lane<YW, XO, TH, MP, ST> {
  using L = Lane<YW, XO, TH, MP, ST>;
  using typename L::Own;
  using typename L::T;
  using L::Tn, L::p, L::k, L::sc, L::e_in, L::ends;
  static constexpr int HR = L::HR;

  __device__ __forceinline__ Tile(const DevParams &p_, const SweepConsts &k_, const T *gs_,
                                  T *gout_, const float *Tin_, float *Tout_,
                                  const StepScalars &sc_, int C0)
      : L(p_, k_, gs_, gout_, Tin_, Tout_, sc_, C0) {}

  // temperature field values of the rows below and above row r: on adiabatic wall columns the
  // ghost copies the row itself
  __device__ __forceinline__ void mirror(int r, V c, V &dn, V &up) const {
    if (YW && !XO && p.adiabatic) {
      if (r == 0) this->mirror_bottom(dn, c);
      if (r == p.ny - 1) {
        if (wall_adiabatic(p, this->x0, true)) up.x = c.x;
        if (wall_adiabatic(p, this->x0 + this->o1, true)) up.y = c.y;
      }
    }
  }

  // the tile with output rows [Y0, ye), at most MAXW - 2 HR of them
  __device__ __forceinline__ void run(int Y0, int ye, TileSmem<MAXW> &S) {
    // (through the shuffle the warp's row is one value to the compiler, its tests branches
    // of the whole warp)
    const int w = __shfl_sync(kAll, (int)(threadIdx.x >> 5), 0), lane = (int)(threadIdx.x & 31);
    const int r = Y0 - HR + w, n = ye - Y0 + 2 * HR;
    const bool solid = YW && (unsigned)r >= (unsigned)p.ny;
    const bool out = r >= Y0 && r < ye;
    V m[9], psi = vdup(0.0f), T0 = vdup(0.0f), cfx, cfz;
    // ---------------- phase 0 ----------------
    if (w < n) {
      if (solid) {
        if (TH) T0 = this->wall_T(r, T0);
      } else {
        this->load_row(true, r);
        if (XO && ends) this->open_ends(r);
        T0 = Tn;
        this->moments(m);
        bool neg0 = false, neg1 = false;
        this->state(m[0], T0, psi, cfx, cfz, neg0, neg1);
        V dr = m[0], dt = T0;
        if (XO && ends) {  // (a ghost's populations include unfixed placeholders)
          if (this->ghost(0)) {
            dr.x = dt.x = 0.0f;
            neg0 = false;
          }
          if (this->ghost(1)) {
            dr.y = dt.y = 0.0f;
            neg1 = false;
          }
        }
        this->track(dr, dt, neg0 || neg1);
      }
      if (MP) S.a[w][lane] = psi;
      if (TH) S.t[w][lane] = T0;
    }
    __syncthreads();
    // ---------------- phase 1 ----------------
    V u_x = vdup(0.0f), u_y = vdup(0.0f), cl = vdup(0.0f);
    if (w >= 1 && w < n - 1 && !solid) {
      V dn = vdup(0.0f), up = vdup(0.0f), Fx, Fy, fm2;
      if (MP) {
        dn = S.a[w - 1][lane];
        up = S.a[w + 1][lane];
      }
      this->forces(r, YW && (r == 0 || r == p.ny - 1), dn, psi, up, T0, m[0], Fx, Fy, fm2);
      const V rho = kp(k.rho_ref) + m[0];
      const V ir = vrcp(rho);
      const V jx = vfma(kl(0.5f), Fx, m[3]), jy = vfma(kl(0.5f), Fy, m[5]);  // rho u
      u_x = jx * ir;
      u_y = jy * ir;
      if (TH) cl = k1(k.lam23_cv) * ir;
      if (out) this->collide_store(r, m, rho, jx, jy, u_x, u_y, Fx, Fy, fm2);
      if (TH && XO && e_in) {
        // the velocity inlet's ghost holds the inlet velocity
        u_x = this->inlet_set(u_x, sc.u_in);
        u_y = this->inlet_set(u_y, 0.0f);
      }
    }
    if (!TH) return;
    S.b[w][lane] = u_x;
    S.c[w][lane] = u_y;
    __syncthreads();
    // ---------------- phase 2 ----------------
    V acc, v;
    Own o;
    if (w >= 2 && w < n - 2) {
      if (solid) {
        v = T0;
      } else {
        V dn = S.t[w - 1][lane], up = S.t[w + 1][lane];
        mirror(r, T0, dn, up);
        o = this->own_values(S.b[w - 1][lane], u_x, S.b[w + 1][lane], S.c[w - 1][lane], u_y,
                             S.c[w + 1][lane], cl, T0, cfx, cfz);
        acc = this->rate(dn, T0, up, o);
        v = vfma(kl(0.5f), acc, T0);
      }
      S.a[w][lane] = v;
    }
    __syncthreads();
    // ---------------- phases 3 and 4 ----------------
    if (w >= 3 && w < n - 3) {
      if (!solid) {
        V dn = S.a[w - 1][lane], up = S.a[w + 1][lane];
        mirror(r, v, dn, up);
        const V h = this->rate(dn, v, up, o);
        acc = vfma(kl(2.0f), h, acc);
        v = vfma(kl(0.5f), h, T0);
      }
      S.b[w][lane] = v;
    }
    __syncthreads();
    if (w >= 4 && w < n - 4) {
      if (!solid) {
        V dn = S.b[w - 1][lane], up = S.b[w + 1][lane];
        mirror(r, v, dn, up);
        const V h = this->rate(dn, v, up, o);
        acc = vfma(kl(2.0f), h, acc);
        v = T0 + h;
      }
      S.a[w][lane] = v;
    }
    __syncthreads();
    // ---------------- phase 5 ----------------
    if (out) {
      V dn = S.a[w - 1][lane], up = S.a[w + 1][lane];
      mirror(r, v, dn, up);
      const V h = this->rate(dn, v, up, o);
      this->store_T(r, vfma(k1(1.0f / 6.0f), acc + h, T0));
    }
  }
};

}  // namespace

}  // namespace lbm
