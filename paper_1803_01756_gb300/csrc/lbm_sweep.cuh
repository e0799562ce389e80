// Fused lattice update by independent warps: the sweep that the single-lattice kernel
// (lbm_sweep_launch.cuh) and the batched one (lbm_sweep_batch.cuh) share.
//
// A warp owns a strip of 64 lattice columns (two adjacent columns per lane, the first one
// even) and a chunk of rows, and sweeps the rows upward.  What a node needs from other rows
// stays in the lane's registers, but for the values that a node's own RK4 stages share over
// four row steps: those are in a ring in shared memory that only the lane itself reads (6 KB a
// warp).  What it needs from other columns comes from the neighbouring lanes by shuffles.  So
// there is no barrier, and the warps of an SM drift freely past one another.  Per swept row r:
//   S0 row r   : pull-streaming with boundary rules (Eq. 12), moments, density (Eq. 13),
//                pseudopotential deviation (Eqs. 10-11)
//   S1 row r-1 : forces (Eqs. 9, 14, 15), velocity (Eq. 13), MRT collision with Li forcing
//                (Eqs. 6-8) and the store of the populations
//   S2 row r-2 : div u and the first RK4 slope h1 of Eq. 16 (Eq. 18)
//   S3 row r-3 : h2      S4 row r-4 : h3      S5 row r-5 : h4 and Eq. 17
// The lane's arithmetic is in lbm_lane.cuh.  With the energy equation 5 rows below and above
// the chunk are swept too, without it one.
#pragma once

#include "lbm_lane.cuh"

namespace lbm {

namespace {

// One warp's sweep: the strip with first column C0, output rows [Y0, ye).
template <bool YW, bool XO, bool TH, bool MP, class ST>
struct Sweep : Lane<YW, XO, TH, MP, ST> {
  using L = Lane<YW, XO, TH, MP, ST>;
  using typename L::Own;
  using typename L::T;
  using L::g, L::Tn, L::p, L::k, L::c0, L::sc, L::e_in, L::e_out, L::ends;
  static constexpr int HR = L::HR;
  static constexpr int NW = HR > 2 ? HR : 2;  // lowest row r whose step reaches no wall below

  int Y0, ye;
  unsigned span;          // rows NW .. NW + span - 1 are away from the walls
  // Carried from row step to row step; an array of two is indexed by the parity of the
  // row's step, so that with two steps per loop iteration few values are copied.
  V m[2][9];              // moments of a row
  V psi[2];               // psi - psi_r
  V cfx[2], cfz[2], cl;   // energy coefficients
  V ux[2], uy[2];
  V T1, T2, T3;           // T of the three newest finished rows
  V K2[2], K3[2], K4[2];  // RK stage fields
  V acc1, acc2, acc3;     // sums h1, h1 + 2 h2, h1 + 2 h2 + 2 h3 of three rows
  float4 *own_s;          // the lane's slots in the warp's ring of four rows: [row][3][32]

  __device__ __forceinline__ Sweep(const DevParams &p_, const SweepConsts &k_, const T *gs_,
                                   T *gout_, const float *Tin_, float *Tout_,
                                   const StepScalars &sc_, int C0, int Y0_, int ye_,
                                   float4 *ring)
      : L(p_, k_, gs_, gout_, Tin_, Tout_, sc_, C0), Y0(Y0_), ye(ye_) {
    own_s = ring + (threadIdx.x & 31);
    span = (unsigned)max(0, p.ny - 2 - NW);
    const V z = vdup(0.0f);
#pragma unroll
    for (int i = 0; i < 9; i++) m[0][i] = m[1][i] = z;
#pragma unroll
    for (int i = 0; i < 2; i++)
      psi[i] = cfx[i] = cfz[i] = ux[i] = uy[i] = K2[i] = K3[i] = K4[i] = z;
    cl = T1 = T2 = T3 = acc1 = acc2 = acc3 = z;
  }

  // the ghosts of row q of a new stage field v; below: the field's row q - 1
  __device__ __forceinline__ V stage_ghosts(bool near, int q, V v, V &below) const {
    if (near) {
      if ((unsigned)q >= (unsigned)p.ny) v = this->wall_T(q, below);
      if (!XO && q == 0) this->mirror_bottom(below, v);
    }
    return v;
  }

  __device__ __forceinline__ void put_own(int j, const Own &o) {
    float4 *d = own_s + (j & 3) * 96;
    d[0] = make_float4(o.nux.x, o.nux.y, o.nuy.x, o.nuy.y);
    d[32] = make_float4(o.cl.x, o.cl.y, o.Tb.x, o.Tb.y);
    d[64] = make_float4(o.nE1.x, o.nE1.y, o.nE2.x, o.nE2.y);
  }
  __device__ __forceinline__ Own get_own(int j) const {
    const float4 *d = own_s + (j & 3) * 96;
    const float4 a = d[0], b = d[32], c = d[64];
    return Own{vset(a.x, a.y), vset(a.z, a.w), vset(b.x, b.y),
               vset(b.z, b.w), vset(c.x, c.y), vset(c.z, c.w)};
  }
  // One row step: row r = Y0 - HR + j, P = j & 1.  Every value is computed in the straight
  // line, and a rare case (wall rows, open ends) overwrites it afterwards, so that no value
  // that is carried on has two sources to be copied together.
  template <int P, bool WARM>
  __device__ __forceinline__ void step(const int j, const int J) {
    constexpr int Q = 1 - P;
    const int r = Y0 - HR + j;
    const unsigned uny = (unsigned)p.ny;
    // one of the step's rows (r + 1 down to r - HR) is a wall row or next to one
    const bool near = YW && (unsigned)(r - NW) >= span;
    // ---------------- S0: row r ----------------
    const bool solid = near && (unsigned)r >= uny;
    if (XO && ends && !solid) this->open_ends(r);
    V T_r = Tn;
    this->moments(m[P]);
    const V drho = m[P][0];
    V psi_r = vdup(0.0f), cfx_r, cfz_r;
    bool neg0 = false, neg1 = false;
    this->state(drho, T_r, psi_r, cfx_r, cfz_r, neg0, neg1);
    // (a ghost's populations include unfixed placeholders, a solid row's are left over)
    bool neg = neg0 || neg1;
    V dr = drho, dt = T_r;
    if (XO && ends) {
      if (this->ghost(0)) dr.x = dt.x = 0.0f;
      if (this->ghost(1)) dr.y = dt.y = 0.0f;
      if (MP) neg = (neg0 && !this->ghost(0)) || (neg1 && !this->ghost(1));
    }
    if (near) {
      if (solid) {
        psi_r = dr = dt = vdup(0.0f);
        T_r = this->wall_T(r, T1);
        neg = false;
      }
      if (TH && !XO && r == 0) this->mirror_bottom(T1, T_r);
    }
    this->track(dr, dt, neg);
    if (j + 1 < J) this->load_row(near, r + 1);
    // (keeps the loads here: moved down to the end of the step they are not back in time;
    // 4096 x 512: 53.7 against 64.6 us per update)
    __syncwarp();

    // ---------------- S1: row r-1 (forces, velocity, collision) ----------------
    V u_x = vdup(0.0f), u_y = vdup(0.0f), cl_q = vdup(0.0f);
    if (!WARM || j >= 2) {
      const int q = r - 1;
      const V (&n)[9] = m[Q];
      V Fx, Fy, fm2;
      this->forces(q, near && (q == 0 || q == p.ny - 1), psi[P], psi[Q], psi_r, T1, n[0], Fx, Fy,
                   fm2);
      const V rho = kp(k.rho_ref) + n[0];
      const V ir = vrcp(rho);
      const V jx = vfma(kl(0.5f), Fx, n[3]), jy = vfma(kl(0.5f), Fy, n[5]);  // rho u
      u_x = jx * ir;
      u_y = jy * ir;
      if (TH) cl_q = k1(k.lam23_cv) * ir;
      if ((unsigned)(q - Y0) < (unsigned)(ye - Y0))
        this->collide_store(q, n, rho, jx, jy, u_x, u_y, Fx, Fy, fm2);
      if (TH) {
        // the velocity inlet's ghost holds the inlet velocity
        if (XO && e_in) {
          u_x = this->inlet_set(u_x, sc.u_in);
          u_y = this->inlet_set(u_y, 0.0f);
        }
        if (near && (unsigned)q >= uny) u_x = u_y = vdup(0.0f);
      }
    }
    if (TH) {
      if (!WARM || j >= 4) {
        // ---------------- S2: row r-2 (div u, h1) ----------------
        const Own o = this->own_values(ux[Q], ux[P], u_x, uy[Q], uy[P], u_y, cl, T2, cfx[P], cfz[P]);
        put_own(j, o);
        const V h1 = this->rate(T3, T2, T1, o);
        const V v2 = stage_ghosts(near, r - 2, vfma(kl(0.5f), h1, T2), K2[Q]);
        if (!WARM || j >= 6) {
          // ---------------- S3: row r-3 (h2) ----------------
          const Own o3 = get_own(j - 1);
          const V h2 = this->rate(K2[P], K2[Q], v2, o3);
          const V v3 = stage_ghosts(near, r - 3, vfma(kl(0.5f), h2, o3.Tb), K3[P]);
          if (!WARM || j >= 8) {
            // ---------------- S4: row r-4 (h3) ----------------
            const Own o4 = get_own(j - 2);
            const V h3 = this->rate(K3[Q], K3[P], v3, o4);
            const V v4 = stage_ghosts(near, r - 4, o4.Tb + h3, K4[Q]);
            if (!WARM) {
              // ---------------- S5: row r-5 (h4, new temperature) ----------------
              const Own o5 = get_own(j - 3);
              const V h4 = this->rate(K4[P], K4[Q], v4, o5);
              const V Tnew = vfma(k1(1.0f / 6.0f), acc3 + h4, o5.Tb);
              this->store_T(r - 5, Tnew);
            }
            acc3 = vfma(kl(2.0f), h3, acc2);
            K4[P] = vcopy(v4);
          }
          acc2 = vfma(kl(2.0f), h2, acc1);
          K3[Q] = vcopy(v3);
        }
        acc1 = vcopy(h1);
        K2[P] = vcopy(v2);
      }
      ux[Q] = vcopy(u_x);
      uy[Q] = vcopy(u_y);
      cl = vcopy(cl_q);
      cfx[P] = vcopy(cfx_r);
      cfz[P] = vcopy(cfz_r);
      T3 = vcopy(T2);
      T2 = vcopy(T1);
    }
    psi[P] = vcopy(psi_r);
    T1 = vcopy(T_r);
  }

  __device__ __forceinline__ void run(unsigned *status) {
    const int J = ye - Y0 + 2 * HR;
    constexpr int JW = 2 * HR;  // steps until every stage has a row (even, below J)
    this->load_row(true, Y0 - HR);
#pragma unroll 1
    for (int j = 0; j < JW; j += 2) {
      step<0, true>(j, J);
      step<1, true>(j + 1, J);
    }
#pragma unroll 1
    for (int j = JW;;) {
      step<0, false>(j, J);
      if (++j >= J) break;
      step<1, false>(j, J);
      if (++j >= J) break;
    }
    this->finish(status);
  }
};

}  // namespace

}  // namespace lbm
