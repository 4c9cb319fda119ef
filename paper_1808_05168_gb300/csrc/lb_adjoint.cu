// lb_adjoint.cu -- reverse-mode (adjoint) sweep of the fluctuating LB step for the gradient of
// the time-averaged mean-pressure shift
//     L = (1/T) sum_{t<T} Pbar(t) |_{kT}  -  (1/T) sum_{t<T} Pbar(t) |_{kT = 0}
// with respect to (G, lambda_s, lambda_d), on a fixed noise stream, both runs from the rest
// state.  Pbar(t) is the spatial mean of the mechanical pressure (Sec. III.C) of the
// pre-collision state of step t.
//
// One step k maps the stored state f*_{k-1} to f*_k (Eq. LB with Eq. MRT).  Its adjoint maps
// fbar*_k (the loss's sensitivity to f*_k) to fbar*_{k-1} and adds the step's share of the
// parameter gradient, in three passes:
//   1. densities: rho^S of the pre-collision state at every site (needed by the neighbours),
//      computed by the previous adjoint step's gather/push, or on their own at the top of a
//      checkpoint segment;
//   2. local: at every site, the forward quantities are recomputed and the transposed Jacobian
//      of the site update is applied to fbar*_k(r) (plus the pressure term of the loss); this
//      gives the sensitivity to the 18 pulled populations through the site's own moments and
//      densities, the sensitivity to the two neighbour sums sum_l w_l c_l rho^S(r + c_l) of
//      Eq. (aNI), and the parameter contributions;
//   3. gather/push: each site collects what its neighbours' forces and pressures owe to its
//      densities (wall ghosts copy the adjacent row, Sec. II.A), adds it to every pulled
//      population of the species, and pushes the result back along the streaming map (the
//      transpose of the pull with mid-way bounce-back is a one-to-one scatter).
// The forward states are recomputed segment by segment from checkpoints (every C steps) into a
// ring of C states, so memory is O(T/C + C) states.  Passes 2 and 3 come twice: arranged for the
// default options, and with every option.
//
// Supported: every lattice of a batch at once, each with its own loss and gradient; the a*
// correction on or off, wall ghosts copying the adjacent row or taking the fixed wall
// composition, hom or loc noise; both precisions.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "lb_adjoint.cuh"

namespace lbk {

namespace {

// v_l = sum_a T_al m_a (the transpose of the moment transform), Table I.
template <class real>
__device__ __forceinline__ void transpose_moments(const real m[9], real v[9]) {
  const real b4 = m[0] + m[3] - 4 * m[8], b5 = m[0] + 4 * m[3] + 8 * m[8];
  v[0] = m[0] - 2 * m[3] + 2 * m[8];
  v[1] = b4 + m[1] + m[4] - m[6];
  v[2] = b4 + m[2] - m[4] - m[7];
  v[3] = b4 - m[1] + m[4] + m[6];
  v[4] = b4 - m[2] - m[4] + m[7];
  v[5] = b5 + m[1] + m[2] + m[5] + 2 * m[6] + 2 * m[7];
  v[6] = b5 - m[1] + m[2] - m[5] - 2 * m[6] + 2 * m[7];
  v[7] = b5 - m[1] - m[2] + m[5] - 2 * m[6] - 2 * m[7];
  v[8] = b5 + m[1] - m[2] - m[5] + 2 * m[6] - 2 * m[7];
}

// m_a = sum_l T_al v_l, Table I (all nine moments).
template <class real>
__device__ __forceinline__ void all_moments(const real v[9], real m[9]) {
  const real a57 = v[5] - v[7], a68 = v[6] - v[8], d13 = v[1] - v[3], d24 = v[2] - v[4];
  const real s13 = v[1] + v[3], s24 = v[2] + v[4], s57 = v[5] + v[7], s68 = v[6] + v[8];
  const real e = s13 + s24, dg = s57 + s68;
  m[0] = v[0] + e + dg;
  m[1] = d13 + a57 - a68;
  m[2] = d24 + a57 + a68;
  m[3] = -2 * v[0] + e + 4 * dg;
  m[4] = s13 - s24;
  m[5] = s57 - s68;
  m[6] = -d13 + 2 * (a57 - a68);
  m[7] = -d24 + 2 * (a57 + a68);
  m[8] = 2 * v[0] - 4 * e + 8 * dg;
}

// The lattice velocities enter through LB_CX / LB_CZ / LB_OPP in fully unrolled loops: as
// compile-time constants, the products with c = 0 and c = +-1 cost no FP64 instruction.

// Deviations of the 9 populations of species s pulled at (x, z) (Eq. LB; reflected at the walls;
// the background streaming shift on non-reflected links), as in the forward kernel.
template <class real>
__device__ __forceinline__ void pull9(const real* __restrict__ f, int Lx, int Lz, int x, int z, double k9, double k36,
                                      int s, double v[9]) {
  const int LzLx = Lx * Lz;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int zs = z - LB_CZ(l);
    const int xs = LB_CX(l) == 0 ? x : (x - LB_CX(l) + Lx) % Lx;
    double val;
    if (zs >= 0 && zs < Lz) {
      val = (double)f[state_index(s, l, zs, xs, Lx, LzLx)];
      if (LB_CZ(l) != 0) {  // the background shift -c_lz w_l rho_bar d_z c_0 (k9, k36: species A)
        const double q = l <= 4 ? k9 : k36;
        const double sh = LB_CZ(l) > 0 ? -q : q;
        val += s == 0 ? sh : -sh;
      }
    } else {
      val = (double)f[state_index(s, LB_OPP(l), z, x, Lx, LzLx)];
    }
    v[l] = val;
  }
}

// Both species: v[9 s + l].
template <class real>
__device__ __forceinline__ void pull18(const real* __restrict__ f, int Lx, int Lz, int x, int z, double k9, double k36,
                                       double v[18]) {
  pull9(f, Lx, Lz, x, z, k9, k36, 0, v);
  pull9(f, Lx, Lz, x, z, k9, k36, 1, v + 9);
}

// Absolute pre-collision densities of site i = z Lx + x of state f, into rho[i] and rho[N + i].
template <class real>
__device__ __forceinline__ void site_densities(const real* __restrict__ f, const LatticeDev<real>& L,
                                               const RowConst<real>* rows, int i, int x, int z, double* rho) {
  const int N = L.Lx * L.Lz;
  double v[18];
  pull18(f, L.Lx, L.Lz, x, z, (double)L.k9, (double)L.k36, v);
  double a = 0, b = 0;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    a += v[l];
    b += v[9 + l];
  }
  rho[i] = (double)rows[z].bgA + a;
  rho[N + i] = (double)rows[z].bgB + b;
}

// The lattice of this block (AdjMap) and the block's first site within it.
__device__ __forceinline__ int adj_lattice(const AdjMap& map) { return map.lat_of[blockIdx.x]; }
__device__ __forceinline__ int adj_site(const AdjMap& map, int li) {
  return (blockIdx.x - map.first[li]) * blockDim.x + threadIdx.x;
}

// Absolute pre-collision densities of every site of every lattice.
template <class real>
__global__ void adj_rho_kernel(const real* __restrict__ f, const LatticeDev<real>* lat, const RowConst<real>* rows,
                               const AdjMap map, double* __restrict__ rho) {
  const int li = adj_lattice(map);
  const LatticeDev<real> L = lat[li];
  const int N = L.Lx * L.Lz;
  const int i = adj_site(map, li);
  if (i >= N) return;
  site_densities(f + L.f_off, L, rows + L.row_off, i, i % L.Lx, i / L.Lx, rho + 2 * L.site_off);
}

// Density of species s at (x, z), beyond a wall the ghost of Sec. II.A: a copy of the adjacent
// row, or (fixed) that row's total density split by the wall composition cw of that row.
template <class real>
__device__ __forceinline__ double rho_at(const double* rho, const RowConst<real>* rows, bool fixed, int Lx, int Lz,
                                         int s, int x, int z) {
  x = (x + Lx) % Lx;
  if (z >= 0 && z < Lz) return rho[s * Lx * Lz + z * Lx + x];
  const int za = z < 0 ? 0 : Lz - 1;
  if (!fixed) return rho[s * Lx * Lz + za * Lx + x];
  const double cw = (double)rows[za].ghost_cA, t = rho[za * Lx + x] + rho[Lx * Lz + za * Lx + x];
  return s == 0 ? cw * t : (1 - cw) * t;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The fourteen normals of a site, exactly those of the forward kernel of the state's precision.
template <class real>
__device__ __forceinline__ void normals14(uint32_t site, uint32_t step, const LatticeDev<real>& L,
                                          const NormalTables* tab, real n[14]) {
  U4 w[4];
  philox_site(site, step, L.lattice_id, L.key0, L.key1, w);
  const uint32_t k[16] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w,
                          w[2].x, w[2].y, w[2].z, w[2].w, w[3].x, w[3].y, w[3].z, w[3].w};
#pragma unroll
  for (int p = 0; p < 7; ++p) normal_pair<real>(k[2 * p], k[2 * p + 1], n[2 * p], n[2 * p + 1], tab);
}

// The local part of the transposed step at every site of every lattice (see the file comment).
// alpha = sign w_loss: weight of the site's pressure in the loss.  Outputs, per lattice at its
// site offset: fl[18][N] (local sensitivity of the pulled
// populations), sb[4][N] (sensitivity of sum_l w_l c_l rho^A, rho^B (r + c_l): x, z for A then
// B), and per block the three parameter partials (G, lambda_s, lambda_d), added to the block's own
// slot of `partials` (zeroed before the sweep; one fixed summation order, step after step).
// The state may be single precision (FP32 deviations); the transposed step is evaluated in double
// precision throughout, since the loss is a small difference of two runs' pressures.
template <class real, bool NOISE>
__global__ void adj_local_kernel(const real* __restrict__ f, const double* __restrict__ fbar,
                                 const LatticeDev<real>* lat, const RowConst<real>* rows,
                                 const AdjConst* __restrict__ kcs, const AdjMap map, const double* __restrict__ rho,
                                 uint32_t step, double sign, double* __restrict__ fl, double* __restrict__ sb,
                                 double* __restrict__ partials, const NormalTables* tab) {
  using real_s = real;
  const int li = adj_lattice(map);
  const LatticeDev<real_s> L = lat[li];
  const AdjConst& kc = kcs[li];
  const double alpha = sign * kc.w_loss;  // weight of this site's pressure in the loss
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz;
  const int i = adj_site(map, li);
  // this lattice's part of the batch's buffers
  f += L.f_off;
  rows += L.row_off;
  fbar += 18 * L.site_off;
  rho += 2 * L.site_off;
  fl += 18 * L.site_off;
  sb += 4 * L.site_off;
  double gG = 0, gS = 0, gD = 0;
  const bool astar = L.flags & DF_ASTAR, fixed = L.flags & DF_WALL_FIXED, loc = NOISE && (L.flags & DF_NOISE_LOC);
  if (i < N) {
    const int x = i % Lx, z = i / Lx;
    double v[18];
    pull18(f, Lx, Lz, x, z, (double)L.k9, (double)L.k36, v);
    double mA[9], mB[9];
    all_moments(v, mA);
    all_moments(v + 9, mB);
    const double rA = rho[i], rB = rho[N + i];
    const double rho_t = rA + rB, inv = double(1) / rho_t;
    // neighbour sums (Eq. aNI) and the pressure's neighbour sums, copy-rule ghosts
    double sAx = 0, sAz = 0, sBx = 0, sBz = 0, NA = 0, NB = 0;
#pragma unroll
    for (int l = 1; l < 9; ++l) {
      constexpr double w9 = double(1) / 9, w36 = double(1) / 36;
      const double w = l <= 4 ? w9 : w36, wc2 = l <= 4 ? w9 : 2 * w36;  // w_l, w_l |c_l|^2
      const double a = rho_at(rho, rows, fixed, Lx, Lz, 0, x + LB_CX(l), z + LB_CZ(l));
      const double b = rho_at(rho, rows, fixed, Lx, Lz, 1, x + LB_CX(l), z + LB_CZ(l));
      if (LB_CX(l) != 0) {
        sAx += (LB_CX(l) * w) * a;
        sBx += (LB_CX(l) * w) * b;
      }
      if (LB_CZ(l) != 0) {
        sAz += (LB_CZ(l) * w) * a;
        sBz += (LB_CZ(l) * w) * b;
      }
      NA += wc2 * a;
      NB += wc2 * b;
    }
    const double G = L.G;
    const double FNx = -G * (rA * sBx + rB * sAx), FNz = -G * (rA * sBz + rB * sAz);
    const double cA = rA * inv, cB = rB * inv;
    const double ne = rho_t * L.g3;
    // the species' forces: with a*, F^S = (rho^S / rho) F_N; without, F^A = -G rho^A s^B and
    // F^B = -G rho^B s^A; plus the gradient forcing +- (0, rho g3)
    const double FA[2] = {astar ? cA * FNx : -G * rA * sBx, (astar ? cA * FNz : -G * rA * sBz) + ne};
    const double FB[2] = {astar ? cB * FNx : -G * rB * sAx, (astar ? cB * FNz : -G * rB * sAz) - ne};
    const double Px = mA[1] + mB[1] + double(0.5) * FNx, Pz = mA[2] + mB[2] + double(0.5) * FNz;
    const double Ux = Px * inv, Uz = Pz * inv;
    const double ld = L.lam[1], le = L.lam[3], ls = L.lam[4], lq = L.lam[6], leps = L.lam[8];
    const double lam[9] = {double(1), ld, ld, le, ls, ls, lq, lq, leps};

    double n[14];
    if (NOISE) {
      real_s nn[14];
      normals14<real_s>((uint32_t)i, step, L, tab, nn);
#pragma unroll
      for (int q = 0; q < 14; ++q) n[q] = (double)nn[q];
    }

    // adjoints accumulated over both species
    double Ubx = 0, Ubz = 0, FNbx = 0, FNbz = 0, rhob_t = 0, invb = 0;
    double rhob[2] = {0, 0};
    double mb[2][9];
    double lamb_d = 0, lamb_s = 0;
    double sbarA[9], sbarB[9];
    double Fb[2][2];  // sensitivities of the species' forces (without a*)
    for (int s = 0; s < 2; ++s) {
      const double* m = s == 0 ? mA : mB;
      const double rs = s == 0 ? rA : rB;
      const double* F = s == 0 ? FA : FB;
      double g[9];
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        const double w = l == 0 ? double(4) / 9 : (l <= 4 ? double(1) / 9 : double(1) / 36);
        g[l] = w * fbar[(s * 9 + l) * N + i];
      }
      double sbar[9];
      all_moments(g, sbar);  // sbar_a = (1/N_a) sum_l T_al w_l fbar_l, before the 1/N_a
      const double invN[9] = {1, 3, 3, double(0.25), double(2.25), 9, double(1.5), double(1.5), double(0.0625)};
#pragma unroll
      for (int a = 0; a < 9; ++a) sbar[a] *= invN[a];
      for (int a = 0; a < 9; ++a) (s == 0 ? sbarA : sbarB)[a] = sbar[a];
      // s_0 = rho^S
      rhob[s] += sbar[0];
      // equilibrium moments and forcing sources
      const double UxUx = Ux * Ux, UzUz = Uz * Uz;
      const double meq[6] = {0, rs * Ux, rs * Uz, 3 * rs * (UxUx + UzUz), rs * (UxUx - UzUz), rs * Ux * Uz};
      const double src[6] = {0, F[0], F[1], 6 * (Ux * F[0] + Uz * F[1]), 2 * (Ux * F[0] - Uz * F[1]),
                           Ux * F[1] + Uz * F[0]};
      double mbar[9];
      mbar[0] = 0;
      double meqb[6], srcb[6];
      for (int a = 1; a < 9; ++a) mbar[a] = kc.oml[a] * sbar[a];
      for (int a = 1; a < 6; ++a) {
        meqb[a] = lam[a] * sbar[a];
        srcb[a] = kc.ohl[a] * sbar[a];
        const double dl = sbar[a] * (meq[a] - m[a] - double(0.5) * src[a]);
        if (a <= 2) lamb_d += dl;
        else if (a >= 4) lamb_s += dl;
      }
      // meq -> rho^S, U
      rhob[s] += meqb[1] * Ux + meqb[2] * Uz + 3 * meqb[3] * (UxUx + UzUz) + meqb[4] * (UxUx - UzUz) +
                 meqb[5] * Ux * Uz;
      Ubx += meqb[1] * rs + 6 * meqb[3] * rs * Ux + 2 * meqb[4] * rs * Ux + meqb[5] * rs * Uz;
      Ubz += meqb[2] * rs + 6 * meqb[3] * rs * Uz - 2 * meqb[4] * rs * Uz + meqb[5] * rs * Ux;
      // sources -> F^S, U
      const double Fbx = srcb[1] + 6 * srcb[3] * Ux + 2 * srcb[4] * Ux + srcb[5] * Uz;
      const double Fbz = srcb[2] + 6 * srcb[3] * Uz - 2 * srcb[4] * Uz + srcb[5] * Ux;
      Ubx += 6 * srcb[3] * F[0] + 2 * srcb[4] * F[0] + srcb[5] * F[1];
      Ubz += 6 * srcb[3] * F[1] - 2 * srcb[4] * F[1] + srcb[5] * F[0];
      if (astar) {  // F^S = (rho^S / rho) F_N +- (0, rho g3)
        const double cS = s == 0 ? cA : cB;
        FNbx += cS * Fbx;
        FNbz += cS * Fbz;
        const double cSb = Fbx * FNx + Fbz * FNz;
        rhob[s] += cSb * inv;
        invb += cSb * rs;
      } else {
        Fb[s][0] = Fbx;
        Fb[s][1] = Fbz;
      }
      rhob_t += (s == 0 ? 1 : -1) * L.g3 * Fbz;
      for (int a = 0; a < 9; ++a) mb[s][a] = mbar[a];
    }
    // U = (j^A + j^B + F_N / 2) / rho
    const double Pbx = Ubx * inv, Pbz = Ubz * inv;
    invb += Ubx * Px + Ubz * Pz;
    mb[0][1] += Pbx;
    mb[0][2] += Pbz;
    mb[1][1] += Pbx;
    mb[1][2] += Pbz;
    FNbx += double(0.5) * Pbx;
    FNbz += double(0.5) * Pbz;
    // F_N = -G (rho^A s^B + rho^B s^A)
    gG += (double)(-(FNbx * (rA * sBx + rB * sAx) + FNbz * (rA * sBz + rB * sAz)));
    rhob[0] += -G * (FNbx * sBx + FNbz * sBz);
    rhob[1] += -G * (FNbx * sAx + FNbz * sAz);
    double eAx = 0, eAz = 0, eBx = 0, eBz = 0;  // the species' own forces (without a*)
    if (!astar) {
      gG += -(Fb[0][0] * rA * sBx + Fb[0][1] * rA * sBz + Fb[1][0] * rB * sAx + Fb[1][1] * rB * sAz);
      rhob[0] += -G * (Fb[0][0] * sBx + Fb[0][1] * sBz);
      rhob[1] += -G * (Fb[1][0] * sAx + Fb[1][1] * sAz);
      eAx = -G * rB * Fb[1][0];
      eAz = -G * rB * Fb[1][1];
      eBx = -G * rA * Fb[0][0];
      eBz = -G * rA * Fb[0][1];
    }
    sb[0 * N + i] = -G * rB * FNbx + eAx;  // sensitivity of s^A (x, z)
    sb[1 * N + i] = -G * rB * FNbz + eAz;
    sb[2 * N + i] = -G * rA * FNbx + eBx;  // sensitivity of s^B (x, z)
    sb[3 * N + i] = -G * rA * FNbz + eBz;
    // the loss's pressure at this site: (1/2) sum |c|^2 f + (G/4) [rho^A N^B + rho^B N^A]
    rhob[0] += alpha * double(0.25) * G * NB;
    rhob[1] += alpha * double(0.25) * G * NA;
    gG += (double)(alpha * double(0.25) * (rA * NB + rB * NA));
    // inv = 1 / rho, rho = rho^A + rho^B
    rhob_t += -invb * inv * inv;
    rhob[0] += rhob_t;
    rhob[1] += rhob_t;
    // noise amplitudes depend on lambda_d (moments 1, 2) and lambda_s (moments 4, 5); loc noise
    // also on the site's densities: sigma_mom = p_mom sqrt(rho^A rho^B / rho), sigma^S_a = p_a
    // sqrt(rho^S)
    if (NOISE) {
      const double q1 = n[0] * (sbarA[1] - sbarB[1]) + n[1] * (sbarA[2] - sbarB[2]);
      if (loc) {
        const double sm = sqrt(rA * rB * inv), qA = sqrt(rA), qB = sqrt(rB);
        lamb_d += kc.dpm * sm * q1;
        lamb_s += kc.dp4 * (qA * sbarA[4] * n[3] + qB * sbarB[4] * n[9]) +
                  kc.dp5 * (qA * sbarA[5] * n[4] + qB * sbarB[5] * n[10]);
        // d sm / d rho^A = (rho^B / rho)^2 / (2 sm), d sm / d rho^B = (rho^A / rho)^2 / (2 sm)
        const double hm = kc.pm * q1 * inv * inv / (2 * sm);
        double tA = 0, tB = 0;
#pragma unroll
        for (int a = 3; a < 9; ++a) {
          tA += kc.pa[a] * sbarA[a] * n[a - 1];
          tB += kc.pa[a] * sbarB[a] * n[a + 5];
        }
        rhob[0] += hm * rB * rB + tA / (2 * qA);
        rhob[1] += hm * rA * rA + tB / (2 * qB);
      } else {
        lamb_d += kc.dsm * q1;
        lamb_s += kc.d4 * (sbarA[4] * n[3] + sbarB[4] * n[9]) + kc.d5 * (sbarA[5] * n[4] + sbarB[5] * n[10]);
      }
    }
    gS += (double)lamb_s;
    gD += (double)lamb_d;
    // back to the pulled populations: moments (transposed), density (every link), kinetic pressure
    for (int s = 0; s < 2; ++s) {
      double o[9];
      mb[s][0] = rhob[s];
      transpose_moments(mb[s], o);
      const double k1 = alpha * double(0.5), k2 = alpha;  // alpha |c_l|^2 / 2 on the axis, diagonal links
#pragma unroll
      for (int l = 0; l < 9; ++l) fl[(s * 9 + l) * N + i] = l == 0 ? o[l] : o[l] + (l <= 4 ? k1 : k2);
    }
  }
  // block partials of the parameter gradient
  __shared__ double red[3][32];
  gG = warp_sum(gG);
  gS = warp_sum(gS);
  gD = warp_sum(gD);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    red[0][wid] = gG;
    red[1][wid] = gS;
    red[2][wid] = gD;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0, c = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += red[0][w];
      b += red[1][w];
      c += red[2][w];
    }
    partials[3 * blockIdx.x + 0] += a;
    partials[3 * blockIdx.x + 1] += b;
    partials[3 * blockIdx.x + 2] += c;
  }
}

// Gather the neighbour-owed density sensitivities and push along the transposed streaming map.
// With f_next (the state before f_prev) given, also the densities of f_next into rho_next, for the
// next adjoint step (one launch instead of two).  Two threads per site, one per species (blocks of
// 2 kAdjBlock threads over the lattice's adjoint blocks): the species' work is independent but
// for the fixed-composition ghosts, which mix both.
template <class real>
__global__ void adj_gather_push_kernel(const LatticeDev<real>* lat, const RowConst<real>* rows,
                                       const AdjConst* __restrict__ kcs, const AdjMap map,
                                       const double* __restrict__ rho, const double* __restrict__ fl,
                                       const double* __restrict__ sb, double sign, double* __restrict__ fbar_prev,
                                       const real* __restrict__ f_next, double* __restrict__ rho_next) {
  const int li = adj_lattice(map);
  const LatticeDev<real> L = lat[li];
  const double alpha = sign * kcs[li].w_loss;
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz;
  const int t = adj_site(map, li), i = t >> 1, sp = t & 1;  // site, species
  if (i >= N) return;
  rows += L.row_off;
  rho += 2 * L.site_off;
  fl += 18 * L.site_off;
  sb += 4 * L.site_off;
  fbar_prev += 18 * L.site_off;
  if (f_next) f_next += L.f_off;
  rho_next += 2 * L.site_off;
  const int x = i % Lx, z = i / Lx;
  if (f_next) {  // this species' density of f_next at the site
    double v[9];
    pull9(f_next, Lx, Lz, x, z, (double)L.k9, (double)L.k36, sp, v);
    double a = 0;
#pragma unroll
    for (int l = 0; l < 9; ++l) a += v[l];
    rho_next[sp * N + i] = (double)(sp == 0 ? rows[z].bgA : rows[z].bgB) + a;
  }
  const double q = alpha * 0.25 * (double)L.G;
  const bool fixed = L.flags & DF_WALL_FIXED;
  double rb = 0;
#pragma unroll
  for (int l = 1; l < 9; ++l) {
    constexpr double w9 = 1.0 / 9, w36 = 1.0 / 36;
    const double w = l <= 4 ? w9 : w36, wc2 = l <= 4 ? w9 : 2 * w36;  // w_l, w_l |c_l|^2
    // what the site j = (x - c_lx, zs) owes the density of species s its link l reaches: through
    // its neighbour sums of s (sb[2 s], sb[2 s + 1]) and its pressure, which pairs s with the
    // other species' density there
    auto owed = [&](int zs, int s) {
      const int j = zs * Lx + (LB_CX(l) == 0 ? x : (x - LB_CX(l) + Lx) % Lx);
      const double* sx = sb + (2 * s) * N;
      const double* sz = sb + (2 * s + 1) * N;
      double ts = 0;
      if (LB_CX(l) != 0) ts = LB_CX(l) * sx[j];
      if (LB_CZ(l) != 0) ts = LB_CX(l) != 0 ? ts + LB_CZ(l) * sz[j] : LB_CZ(l) * sz[j];
      return w * ts + (wc2 * q) * rho[(1 - s) * N + j];
    };
    const int zs = z - LB_CZ(l);
    if (zs >= 0 && zs < Lz) rb += owed(zs, sp);
    // the wall ghost next to this row: a copy of this row's densities, or (fixed) this row's total
    // density split by the wall composition
    if ((z == 0 && LB_CZ(l) == -1) || (z == Lz - 1 && LB_CZ(l) == 1)) {
      if (fixed) {
        const double cw = (double)rows[z].ghost_cA;
        rb += cw * owed(z, 0) + (1 - cw) * owed(z, 1);
      } else {
        rb += owed(z, sp);
      }
    }
  }
  const int64_t LzLx = N;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const double val = fl[(sp * 9 + l) * N + i] + rb;
    const int zs = z - LB_CZ(l);
    if (zs >= 0 && zs < Lz) {
      const int xs = LB_CX(l) == 0 ? x : (x - LB_CX(l) + Lx) % Lx;
      fbar_prev[(sp * 9 + l) * LzLx + zs * Lx + xs] = val;
    } else {
      fbar_prev[(sp * 9 + LB_OPP(l)) * LzLx + z * Lx + x] = val;
    }
  }
}

// ---- the default options (a*, copy-rule ghosts, hom noise) ----------------------------------------
// The transposed step is bound by the FP64 pipe (two lanes per clock and SM), so these kernels are
// arranged for the fewest FP64 instructions: about 320 per site and step (280 in the local pass, 43 in the
// gather) against about 1000 of the kernels above, which remain for the other options.
//  - what both species share is formed once from their density-weighted sums T_a = sum_s rho^S t^S_a;
//  - with a* the sensitivities of m^eq and of the source act on the same combinations of the moments,
//    so one dot product per species (K_1 .. K_5) gives both shares of rho^S;
//  - the link weights, 1/N_a and the rates are folded into AdjConst;
//  - the moments' sensitivities are handed over (3 per species with unit rates, else 9) and turned
//    into populations by the gather, not written as 18 populations and read again;
//  - what a site's pressure owes its neighbours' densities is, under the copy rule, what they owe it:
//    the local pass adds it twice and the gather has only the forces' share to collect;
//  - the parameters' shares stay per site (one addition each) instead of a warp reduction per step;
//  - FP32 populations are widened by their bits (the conversion instruction runs at the FP64 rate).
// 256 x 128, 500 steps, FP64: 62 -> 52 ms for the whole gradient; eight lattices from FP32 state, 300
// steps: 133 -> 83 ms (the local pass 290 -> 171 us a step, the gather 92 -> 28).

template <class real>
struct PairOfState;
template <>
struct PairOfState<float> {
  using type = float2;
};
template <>
struct PairOfState<double> {
  using type = double2;
};

// The nine pairs pulled at (x, z), as stored (Eq. LB, reflected at the walls).
template <class real>
__device__ __forceinline__ void load_pairs(const real* __restrict__ f, int Lx, int Lz, int x, int z,
                                           typename PairOfState<real>::type w[9]) {
  using P = typename PairOfState<real>::type;
  const P* g = reinterpret_cast<const P*>(f);
  const int N = Lx * Lz, xm = x == 0 ? Lx - 1 : x - 1, xp = x + 1 == Lx ? 0 : x + 1;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int zs = z - LB_CZ(l), xs = LB_CX(l) == 0 ? x : (LB_CX(l) > 0 ? xm : xp);
    const bool in = LB_CZ(l) == 0 || (zs >= 0 && zs < Lz);
    w[l] = g[in ? l * N + zs * Lx + xs : LB_OPP(l) * N + z * Lx + x];
  }
}

// Links 1..8 of both species widened, v[s][l], the wall rows' background shifts applied per link (in
// interior rows they leave every moment but m_2 alone and the caller adds them there; none in FP64).
template <class real>
__device__ __forceinline__ void pull_pairs(const real* __restrict__ f, const LatticeDev<real>& L, int x, int z,
                                           double v[2][9]) {
  typename PairOfState<real>::type w[9];
  const int Lz = L.Lz;
  const bool wall = z == 0 || z == Lz - 1;
  load_pairs<real>(f, L.Lx, Lz, x, z, w);
#pragma unroll
  for (int l = 1; l < 9; ++l) {
    v[0][l] = widen(w[l].x);
    v[1][l] = widen(w[l].y);
    if (sizeof(real) == 4 && LB_CZ(l) != 0 && wall) {
      const int zs = z - LB_CZ(l);
      if (zs >= 0 && zs < Lz) {
        const double q = l <= 4 ? (double)L.k9 : (double)L.k36, sh = LB_CZ(l) > 0 ? -q : q;
        v[0][l] += sh;
        v[1][l] -= sh;
      }
    }
  }
}

// ---- densities and pressures of a segment's states -------------------------------------------------
// The wall rows' shifts on the stored FP32 pairs, as `deviations` of the step kernels.
__device__ __forceinline__ void shift_wall32(float2 w[9], bool below, bool above, float k9, float k36) {
  const float b9 = below ? k9 : 0.f, b36 = below ? k36 : 0.f, a9 = above ? k9 : 0.f, a36 = above ? k36 : 0.f;
  w[2] = make_float2(w[2].x - b9, w[2].y + b9);
  w[4] = make_float2(w[4].x + a9, w[4].y - a9);
  w[5] = make_float2(w[5].x - b36, w[5].y + b36);
  w[6] = make_float2(w[6].x - b36, w[6].y + b36);
  w[7] = make_float2(w[7].x + a36, w[7].y - a36);
  w[8] = make_float2(w[8].x + a36, w[8].y - a36);
}

// Pre-collision densities of every site of the `gridDim.y` states at f, f + S, ..: absolute densities in
// double (rho: [2][N] per lattice at 2 site_off, states 2 NS apart; null: not wanted) and, for FP32, the
// deviations in single precision, summed as the step kernels do (dev: pairs at site_off, NS apart).
template <class real>
__global__ void __launch_bounds__(kAdjBlock)
    adj_density_default(const real* __restrict__ f, int64_t S, const LatticeDev<real>* lat, const RowConst<real>* rows,
                        const AdjMap map, double* __restrict__ rho, float2* __restrict__ dev, int64_t NS) {
  const int li = adj_lattice(map);
  const LatticeDev<real>& L = lat[li];
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz, i = adj_site(map, li);
  if (i >= N) return;
  const int z = i / Lx, x = i - z * Lx, k = blockIdx.y;
  typename PairOfState<real>::type w[9];
  load_pairs<real>(f + k * S + L.f_off, Lx, Lz, x, z, w);
  if constexpr (sizeof(real) == 4) {
    if (z == 0 || z == Lz - 1) {
      // absolute: the shifts of the non-reflected links in double (in interior rows they sum to zero)
      if (rho) {
        const double q = (double)L.k9 + 2 * (double)L.k36, sh = (z > 0 ? -q : 0.0) + (z < Lz - 1 ? q : 0.0);
        double a = sh, b = -sh;
#pragma unroll
        for (int l = 0; l < 9; ++l) {
          a += widen(w[l].x);
          b += widen(w[l].y);
        }
        double* r = rho + 2 * (k * NS + L.site_off) + i;
        r[0] = (double)rows[L.row_off + z].bgA + a;
        r[N] = (double)rows[L.row_off + z].bgB + b;
      }
      shift_wall32(w, z > 0, z < Lz - 1, L.k9, L.k36);
    } else if (rho) {
      double a = 0, b = 0;
#pragma unroll
      for (int l = 0; l < 9; ++l) {
        a += widen(w[l].x);
        b += widen(w[l].y);
      }
      double* r = rho + 2 * (k * NS + L.site_off) + i;
      r[0] = (double)rows[L.row_off + z].bgA + a;
      r[N] = (double)rows[L.row_off + z].bgB + b;
    }
    dev[k * NS + L.site_off + i] =
        make_float2((((w[0].x + w[1].x) + (w[2].x + w[3].x)) + ((w[4].x + w[5].x) + (w[6].x + w[7].x))) + w[8].x,
                    (((w[0].y + w[1].y) + (w[2].y + w[3].y)) + ((w[4].y + w[5].y) + (w[6].y + w[7].y))) + w[8].y);
  } else {
    double* r = rho + 2 * (k * NS + L.site_off) + i;
    r[0] = (((w[0].x + w[1].x) + (w[2].x + w[3].x)) + ((w[4].x + w[5].x) + (w[6].x + w[7].x))) + w[8].x;
    r[N] = (((w[0].y + w[1].y) + (w[2].y + w[3].y)) + ((w[4].y + w[5].y) + (w[6].y + w[7].y))) + w[8].y;
  }
}

// The mechanical pressure of one site (Sec. III.C), minus its row's background in FP32: the arithmetic
// of site_update of the step kernels, in the state's precision.  d: the densities (FP32: deviations) as
// pairs through at(row offset, column).
template <class real, class P, class At>
__device__ __forceinline__ real site_pressure(const P w[9], real G, const RowConst<real>& rc, At at, int Lx, int Lz,
                                              int x, int z) {
  real m3[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    auto v = [&](int l) { return s == 0 ? w[l].x : w[l].y; };
    const real e = (v(1) + v(3)) + (v(2) + v(4)), dg = (v(5) + v(7)) + (v(6) + v(8));
    m3[s] = fma(real(-2), v(0), fma(real(4), dg, e));
  }
  const int xm = x == 0 ? Lx - 1 : x - 1, xp = x + 1 == Lx ? 0 : x + 1;
  const int r0 = z * Lx, ru = min(z + 1, Lz - 1) * Lx, rd = max(z - 1, 0) * Lx;
  const P d = at(r0 + x), wv = at(r0 + xm), e = at(r0 + xp), n = at(ru + x), nw = at(ru + xm), ne = at(ru + xp),
          s = at(rd + x), sw = at(rd + xm), se = at(rd + xp);
  const real kin = (m3[0] + m3[1] + 2 * (d.x + d.y)) * (real(1) / 6);
  const real c9 = real(1) / 9, c18 = real(2) / 36;
  const real NA = fma(c9, (e.x + wv.x) + (n.x + s.x), c18 * ((ne.x + nw.x) + (se.x + sw.x)));
  const real NB = fma(c9, (e.y + wv.y) + (n.y + s.y), c18 * ((ne.y + nw.y) + (se.y + sw.y)));
  const real inter = d.x * (rc.nbB + NB) + rc.bgA * NB + d.y * (rc.nbA + NA) + rc.bgB * NA;
  return kin + real(0.25) * G * inter;
}

// The pressure of the `gridDim.y` states at f, f + S, .. summed over each block's sites:
// part[state][block].
template <class real>
__global__ void __launch_bounds__(kAdjBlock)
    adj_pressure(const real* __restrict__ f, int64_t S, const LatticeDev<real>* lat, const RowConst<real>* rows,
                 const AdjMap map, const double* __restrict__ rho, const float2* __restrict__ dev, int64_t NS,
                 double* __restrict__ part) {
  using P = typename PairOfState<real>::type;
  const int li = adj_lattice(map);
  const LatticeDev<real>& L = lat[li];
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz, i = adj_site(map, li), k = blockIdx.y;
  double p = 0;
  if (i < N) {
    const int z = i / Lx, x = i - z * Lx;
    P w[9];
    load_pairs<real>(f + k * S + L.f_off, Lx, Lz, x, z, w);
    const RowConst<real>& rc = rows[L.row_off + z];
    if constexpr (sizeof(real) == 4) {
      if (z == 0 || z == Lz - 1) shift_wall32(w, z > 0, z < Lz - 1, L.k9, L.k36);
      const float2* d = dev + k * NS + L.site_off;
      p = (double)site_pressure<float>(w, L.G, rc, [&](int j) { return d[j]; }, Lx, Lz, x, z);
    } else {
      const double* d = rho + 2 * (k * NS + L.site_off);
      p = site_pressure<double>(w, L.G, rc, [&](int j) { return make_double2(d[j], d[N + j]); }, Lx, Lz, x, z);
    }
  }
  p = warp_sum(p);
  if (threadIdx.x == 0) part[(int64_t)k * map.n_blocks + blockIdx.x] = p;
}

// out[state * n_lat + lattice]: the sums over the lattices' blocks, in a fixed order (one warp each).
__global__ void adj_sum_pressure(const double* __restrict__ part, const AdjMap map, double* __restrict__ out) {
  const int li = blockIdx.x, k = blockIdx.y, b1 = map.first[li + 1];
  double a = 0;
  for (int b = map.first[li] + threadIdx.x; b < b1; b += 32) a += part[(int64_t)k * map.n_blocks + b];
  a = warp_sum(a);
  if (threadIdx.x == 0) out[(int64_t)k * map.n_lat + li] = a;
}

// fbar (and mom and sb below) may still be written by the grid before this one while this one starts: no
// __restrict__, which with const would let them be read as constant for the whole grid.
// 16 warps per SM (128 registers): eight lattices of 256 x 128 246 us per step, 255 with the 12 that the
// compiler's own 168 registers leave.
template <class real, bool NOISE, bool UNIT>
__global__ void __launch_bounds__(kAdjBlock, 16)
    adj_local_default(const real* __restrict__ f, const double* fbar, const LatticeDev<real>* lat,
                      const AdjConst* __restrict__ kcs, const AdjMap map, const double* __restrict__ rho, uint32_t step,
                      double sign, double* __restrict__ mom, double* __restrict__ sb, double* __restrict__ shares,
                      const NormalTables* tab) {
  constexpr int NM = UNIT ? 3 : 9;
  const int li = adj_lattice(map);
  const LatticeDev<real>& L = lat[li];
  const AdjConst& k = kcs[li];
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz, i = adj_site(map, li);
  if (i >= N) return;
  const int64_t so = L.site_off;
  f += L.f_off;
  fbar += 18 * so;
  rho += 2 * so;
  mom += 18 * so;
  sb += 8 * so;
  shares += 3 * so;
  const int z = i / Lx, x = i - z * Lx;
  const double alpha = sign * k.w_loss;  // weight of this site's pressure in the loss
  const bool wall = z == 0 || z == Lz - 1;

  // moments 1, 2, 4, 5 of both species
  double m1[2], m2[2], m4[2], m5[2];
  {
    double v[2][9];
    pull_pairs<real>(f, L, x, z, v);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const double a57 = v[s][5] - v[s][7], a68 = v[s][6] - v[s][8];
      m1[s] = (v[s][1] - v[s][3]) + (a57 - a68);
      m2[s] = (v[s][2] - v[s][4]) + (a57 + a68);
      m4[s] = (v[s][1] + v[s][3]) - (v[s][2] + v[s][4]);
      m5[s] = (v[s][5] + v[s][7]) - (v[s][6] + v[s][8]);
    }
    if (sizeof(real) == 4 && !wall) {
      const double q = 2 * (double)L.k9 + 4 * (double)L.k36;
      m2[0] -= q;
      m2[1] += q;
    }
  }
  // neighbour sums: X, Z = 36 sum_l w_l c_l rho (Eq. aNI), n18 = 18 sum_l w_l |c_l|^2 rho; copy-rule ghosts
  double r[2], X[2], Z[2], n18[2];
  {
    const int xm = x == 0 ? Lx - 1 : x - 1, xp = x + 1 == Lx ? 0 : x + 1;
    const int zu = min(z + 1, Lz - 1) * Lx, zd = max(z - 1, 0) * Lx, zc = z * Lx;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const double* p = rho + s * N;
      const double e = p[zc + xp], w = p[zc + xm], n = p[zu + x], d = p[zd + x];
      const double ne = p[zu + xp], nw = p[zu + xm], se = p[zd + xp], sw = p[zd + xm];
      const double da = ne - sw, db = nw - se;
      r[s] = p[i];
      X[s] = fma(4.0, e - w, da - db);
      Z[s] = fma(4.0, n - d, da + db);
      n18[s] = fma(2.0, (e + w) + (n + d), (ne + sw) + (nw + se));
    }
  }
  const double G = L.G, Gm = G * (-1.0 / 36.0);
  const double inv = site_reciprocal(r[0] + r[1]);
  const double Tx = fma(r[0], X[1], r[1] * X[0]), Tz = fma(r[0], Z[1], r[1] * Z[0]);
  const double Fx = Gm * Tx, Fz = Gm * Tz;          // F_N
  const double ax = Fx * inv, az = Fz * inv;        // F_N / rho
  const double ne = (r[0] + r[1]) * (double)L.g3;   // gradient forcing, + for A, - for B
  const double Px = fma(0.5, Fx, m1[0] + m1[1]), Pz = fma(0.5, Fz, m2[0] + m2[1]);
  const double Ux = Px * inv, Uz = Pz * inv;
  const double UxUx = Ux * Ux, UzUz = Uz * Uz, UxUz = Ux * Uz, Ud = UxUx - UzUz;
  const double ux = Ux * ax, uz = Uz * az, ap = ux + uz, am = ux - uz, cr = fma(Uz, ax, Ux * az);

  double nz[6];  // the normals of moments 1, 2 and of A's and B's 4, 5
  if (NOISE) {
    real nn[14];
    normals14<real>((uint32_t)i, step, L, tab, nn);
    nz[0] = widen(nn[0]), nz[1] = widen(nn[1]), nz[2] = widen(nn[3]), nz[3] = widen(nn[4]), nz[4] = widen(nn[9]),
    nz[5] = widen(nn[10]);
  }
  // so far only what older launches left: the sensitivities come from the grid before this one, and the
  // next one (launched to overlap as well) may start, all before that grid having ended
  wait_for_previous_grid();
  let_next_grid_start();

  // t_a: the moments of w_l fbar_l up to a factor each (sbar_a = t_0/36, t_1/12, t_2/12, t_3/36, t_4/4,
  // t_5/4, t_6/12, t_7/12, t_8/72 with the 1/N_a of the transposed inverse transform)
  double t[2][9];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    double g[9];
#pragma unroll
    for (int l = 0; l < 9; ++l) g[l] = fbar[(s * 9 + l) * N + i];
    const double s57 = g[5] + g[7], s68 = g[6] + g[8], a57 = g[5] - g[7], a68 = g[6] - g[8];
    const double s13 = g[1] + g[3], s24 = g[2] + g[4], d13 = g[1] - g[3], d24 = g[2] - g[4];
    const double dg = s57 + s68, e = s13 + s24, amm = a57 - a68, app = a57 + a68;
    t[s][0] = fma(16.0, g[0], fma(4.0, e, dg));
    t[s][1] = fma(4.0, d13, amm);
    t[s][2] = fma(4.0, d24, app);
    t[s][3] = fma(-8.0, g[0], e + dg);
    t[s][4] = s13 - s24;
    t[s][5] = s57 - s68;
    if (!UNIT) {
      t[s][6] = fma(-2.0, d13, amm);
      t[s][7] = fma(-2.0, d24, app);
      t[s][8] = fma(4.0, g[0], fma(-2.0, e, dg));
    }
  }
  // shares of rho^S through m^eq and through the source
  const double K1 = fma(k.l1, Ux, k.o1 * ax), K2 = fma(k.l1, Uz, k.o1 * az);
  const double K3 = fma(k.l3, UxUx + UzUz, k.o3 * ap), K4 = fma(k.l4, Ud, k.o4 * am), K5 = fma(k.l4, UxUz, k.o5 * cr);
  double rb[2];
#pragma unroll
  for (int s = 0; s < 2; ++s)
    rb[s] = fma(t[s][5], K5, fma(t[s][4], K4, fma(t[s][3], K3, fma(t[s][2], K2, fma(t[s][1], K1, t[s][0] * (1.0 / 36))))));
  double T[6], d[6];
#pragma unroll
  for (int a = 1; a < 6; ++a) {
    T[a] = fma(r[0], t[0][a], r[1] * t[1][a]);
    d[a] = t[0][a] - t[1][a];
  }
  const double p = (2 * k.l3) * T[3], q = (2 * k.l4) * T[4], rr = k.l4 * T[5];
  const double po = k.o3 * T[3], qo = k.o4 * T[4], ro = k.o5 * T[5];
  const double sp = po + qo, sm = po - qo, k34 = fma(k.o3, d[3], -(k.o4 * d[4])), o5d = k.o5 * d[5];
  const double Ubx = fma(o5d, ne, fma(ro, az, fma(sp, ax, fma(rr, Uz, fma(p + q, Ux, k.l1 * T[1])))));
  const double Ubz = fma(k34, ne, fma(ro, ax, fma(sm, az, fma(rr, Ux, fma(p - q, Uz, k.l1 * T[2])))));
  const double Wx = fma(ro, Uz, fma(sp, Ux, k.o1 * T[1])), Wz = fma(ro, Ux, fma(sm, Uz, k.o1 * T[2]));
  const double Pbx = Ubx * inv, Pbz = Ubz * inv;
  const double FNbx = fma(0.5, Pbx, Wx * inv), FNbz = fma(0.5, Pbz, Wz * inv);
  const double invb = fma(Wx, Fx, fma(Wz, Fz, fma(Ubx, Px, Ubz * Pz)));
  const double rt = fma((double)L.g3, fma(o5d, Ux, fma(k34, Uz, k.o1 * d[2])), -(invb * (inv * inv)));
  const double yx = Gm * FNbx, yz = Gm * FNbz, pg = (alpha * (1.0 / 36)) * G;
  rb[0] += fma(pg, n18[1], fma(yx, X[1], fma(yz, Z[1], rt)));
  rb[1] += fma(pg, n18[0], fma(yx, X[0], fma(yz, Z[0], rt)));
  // sensitivities of the neighbour sums (by 36): (x, z, x + z, z - x) of A, then of B
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double sx = yx * r[1 - s], sz = yz * r[1 - s];
    double* o = sb + (int64_t)(4 * s) * N + i;
    o[0] = sx;
    o[N] = sz;
    o[2 * (int64_t)N] = sx + sz;
    o[3 * (int64_t)N] = sz - sx;
  }
  // the parameters' shares
  const double gG = fma(alpha * (1.0 / 72), fma(r[0], n18[1], r[1] * n18[0]), fma(FNbx, Tx, FNbz * Tz) * (-1.0 / 36));
  double ld = fma(T[1], fma(-0.5, ax, Ux), T[2] * fma(-0.5, az, Uz));
  ld = fma(-0.5 * ne, d[2], ld);
  double ls = fma(T[4], Ud - am, T[5] * fma(-0.5, cr, UxUz));
  ls = fma(ne, fma(Uz, d[4], -0.5 * (Ux * d[5])), ls);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    ld = fma(-t[s][1], m1[s], fma(-t[s][2], m2[s], ld));
    ls = fma(-t[s][4], m4[s], fma(-t[s][5], m5[s], ls));
  }
  if (NOISE) {
    ld = fma(k.dsm, fma(nz[0], d[1], nz[1] * d[2]), ld);
    ls = fma(k.d4, fma(t[0][4], nz[2], t[1][4] * nz[4]), ls);
    ls = fma(k.d5, fma(t[0][5], nz[3], t[1][5] * nz[5]), ls);
  }
  shares[i] += gG;
  shares[N + i] = fma(0.25, ls, shares[N + i]);
  shares[2 * (int64_t)N + i] = fma(1.0 / 12, ld, shares[2 * (int64_t)N + i]);
  // the moments' sensitivities
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    double* o = mom + (int64_t)(NM * s) * N + i;
    o[0] = rb[s];
    o[N] = fma(k.b1, t[s][1], Pbx);
    o[2 * (int64_t)N] = fma(k.b1, t[s][2], Pbz);
    if (!UNIT) {
      o[3 * (int64_t)N] = k.b3 * t[s][3];
      o[4 * (int64_t)N] = k.b4 * t[s][4];
      o[5 * (int64_t)N] = k.b4 * t[s][5];
      o[6 * (int64_t)N] = k.b6 * t[s][6];
      o[7 * (int64_t)N] = k.b6 * t[s][7];
      o[8 * (int64_t)N] = k.b8 * t[s][8];
    }
  }
}

// Gather the forces' share of the neighbours, turn the moments' sensitivities into populations and push
// them along the transposed streaming map.  Two threads per site, one per species, as
// adj_gather_push_kernel.
template <class real, bool UNIT>
__global__ void __launch_bounds__(2 * kAdjBlock)
    adj_push_default(const LatticeDev<real>* lat, const AdjConst* __restrict__ kcs, const AdjMap map,
                     const double* mom, const double* sb, double sign, double* __restrict__ fbar_prev) {
  constexpr int NM = UNIT ? 3 : 9;
  const int li = adj_lattice(map);
  const LatticeDev<real>& L = lat[li];
  const int Lx = L.Lx, Lz = L.Lz, N = Lx * Lz;
  const int t = adj_site(map, li), i = t >> 1, sp = t & 1;  // site, species
  if (i >= N) return;
  const int64_t so = L.site_off;
  const int z = i / Lx, x = i - z * Lx;
  const int xm = x == 0 ? Lx - 1 : x - 1, xp = x + 1 == Lx ? 0 : x + 1;
  const bool wall = z == 0 || z == Lz - 1;
  wait_for_previous_grid();
  let_next_grid_start();
  const double* sx = sb + 8 * so + (int64_t)(4 * sp) * N;
  const double *sz = sx + N, *s5 = sz + N, *s6 = s5 + N;  // x + z, z - x
  double rb;
  if (!wall) {
    const int zc = z * Lx, zu = zc + Lx, zd = zc - Lx;
    rb = fma(4.0, (sx[zc + xm] - sx[zc + xp]) + (sz[zd + x] - sz[zu + x]),
             (s5[zd + xm] - s5[zu + xp]) + (s6[zd + xp] - s6[zu + xm]));
  } else {
    // link by link: the neighbours inside the walls, and through the ghost next to this row (a copy of
    // it) the sites of this row
    rb = 0.0;
#pragma unroll
    for (int l = 1; l < 9; ++l) {
      const int xs = LB_CX(l) == 0 ? x : (LB_CX(l) > 0 ? xm : xp), zs = z - LB_CZ(l);
      auto owed = [&](int zz) {
        const int j = zz * Lx + xs;
        return (l <= 4 ? 4.0 : 1.0) * ((double)LB_CX(l) * sx[j] + (double)LB_CZ(l) * sz[j]);
      };
      if (zs >= 0 && zs < Lz) rb += owed(zs);
      if ((z == 0 && LB_CZ(l) == -1) || (z == Lz - 1 && LB_CZ(l) == 1)) rb += owed(z);
    }
  }
  const double* mo = mom + 18 * so + (int64_t)(NM * sp) * N + i;
  const double alpha = sign * kcs[li].w_loss;
  double o[9];
  if (UNIT) {
    const double m0 = mo[0] + rb, m1 = mo[N], m2 = mo[2 * (int64_t)N];
    const double ma = fma(0.5, alpha, m0), md = m0 + alpha;  // kinetic pressure: alpha |c_l|^2 / 2
    const double hp = m1 + m2, hm = m1 - m2;
    o[0] = m0;
    o[1] = ma + m1;
    o[2] = ma + m2;
    o[3] = ma - m1;
    o[4] = ma - m2;
    o[5] = md + hp;
    o[6] = md - hm;
    o[7] = md - hp;
    o[8] = md + hm;
  } else {
    double m[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) m[a] = mo[(int64_t)a * N];
    m[0] += rb;
    transpose_moments(m, o);
#pragma unroll
    for (int l = 1; l < 9; ++l) o[l] += l <= 4 ? 0.5 * alpha : alpha;
  }
  double* out = fbar_prev + 18 * so;
#pragma unroll
  for (int l = 0; l < 9; ++l) {
    const int zs = z - LB_CZ(l), xs = LB_CX(l) == 0 ? x : (LB_CX(l) > 0 ? xm : xp);
    const bool in = LB_CZ(l) == 0 || (zs >= 0 && zs < Lz);
    out[in ? (sp * 9 + l) * (int64_t)N + zs * Lx + xs : (sp * 9 + LB_OPP(l)) * (int64_t)N + z * Lx + x] = o[l];
  }
}

// grads[3 i + p] = sum over the sites of lattice i of its shares [3][N]: block (i, p), threads strided over the sites, then a fixed tree (deterministic).
template <class real>
__global__ void __launch_bounds__(1024) adj_sum_shares(const double* shares, const LatticeDev<real>* lat, double* grads) {
  const LatticeDev<real>& L = lat[blockIdx.x];
  const int N = L.Lx * L.Lz;
  const double* p = shares + 3 * L.site_off + (int64_t)blockIdx.y * N;
  double a = 0;
  for (int i = threadIdx.x; i < N; i += 1024) a += p[i];
  __shared__ double red[32];
  a = warp_sum(a);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x < 32) {
    a = warp_sum(red[threadIdx.x]);
    if (threadIdx.x == 0) grads[3 * blockIdx.x + blockIdx.y] = a;
  }
}

// grads[3 i + k] = sum over the blocks b of lattice i of partials[3 b + k]: one warp per lattice
// (block i), lanes strided over the blocks, then a fixed butterfly (deterministic).
__global__ void adj_sum_partials(const double* partials, const AdjMap map, double* grads) {
  const int li = blockIdx.x;
  const int b0 = map.first[li], n = map.first[li + 1] - b0;
  partials += 3 * (size_t)b0;
  double* grad = grads + 3 * li;
  double a = 0, b = 0, c = 0;
  for (int k = threadIdx.x; k < n; k += 32) {
    a += partials[3 * k];
    b += partials[3 * k + 1];
    c += partials[3 * k + 2];
  }
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  if (threadIdx.x == 0) {
    grad[0] = a;
    grad[1] = b;
    grad[2] = c;
  }
}

}  // namespace

template <class real>
cudaError_t launch_adjoint_step(const real* f_prev, const real* f_next, const double* fbar, double* fbar_prev,
                                const LatticeDev<real>* lat, const RowConst<real>* rows, const AdjConst* kcs,
                                const AdjMap& map, uint32_t step, bool noise, double sign, bool rho_ready, double* rho,
                                double* rho_next, double* fl, double* sb, double* partials, const NormalTables* tab,
                                cudaStream_t s) {
  const int nb = map.n_blocks;
  if (!rho_ready) adj_rho_kernel<real><<<nb, kAdjBlock, 0, s>>>(f_prev, lat, rows, map, rho);
  if (noise)
    adj_local_kernel<real, true>
        <<<nb, kAdjBlock, 0, s>>>(f_prev, fbar, lat, rows, kcs, map, rho, step, sign, fl, sb, partials, tab);
  else
    adj_local_kernel<real, false>
        <<<nb, kAdjBlock, 0, s>>>(f_prev, fbar, lat, rows, kcs, map, rho, step, sign, fl, sb, partials, tab);
  adj_gather_push_kernel<real>
      <<<nb, 2 * kAdjBlock, 0, s>>>(lat, rows, kcs, map, rho, fl, sb, sign, fbar_prev, f_next, rho_next);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_gradient(const double* partials, const AdjMap& map, double* grads, cudaStream_t s) {
  adj_sum_partials<<<map.n_lat, 32, 0, s>>>(partials, map, grads);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_adjoint_densities(const real* f, int64_t S, int n_states, const LatticeDev<real>* lat,
                                     const RowConst<real>* rows, const AdjMap& map, double* rho, float* dev, int64_t NS,
                                     cudaStream_t s) {
  adj_density_default<real><<<dim3(map.n_blocks, n_states), kAdjBlock, 0, s>>>(f, S, lat, rows, map, rho,
                                                                               reinterpret_cast<float2*>(dev), NS);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_adjoint_pressures(const real* f, int64_t S, int n_states, const LatticeDev<real>* lat,
                                     const RowConst<real>* rows, const AdjMap& map, const double* rho, const float* dev,
                                     int64_t NS, double* part, double* out, cudaStream_t s) {
  adj_pressure<real><<<dim3(map.n_blocks, n_states), kAdjBlock, 0, s>>>(
      f, S, lat, rows, map, rho, reinterpret_cast<const float2*>(dev), NS, part);
  adj_sum_pressure<<<dim3(map.n_lat, n_states), 32, 0, s>>>(part, map, out);
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_adjoint_step_default(const real* f_prev, const double* fbar, double* fbar_prev,
                                        const LatticeDev<real>* lat, const AdjConst* kcs, bool unit, const AdjMap& map,
                                        uint32_t step, bool noise, double sign, const double* rho, double* mom, double* sb,
                                        double* shares, const NormalTables* tab, cudaStream_t s) {
  const int nb = map.n_blocks;
  auto pair = [&](auto noise_c, auto unit_c) {
    constexpr bool U = decltype(unit_c)::value;
    launch_overlapped(true, adj_local_default<real, decltype(noise_c)::value, U>, dim3(nb), kAdjBlock, 0, s, f_prev, fbar, lat,
                      kcs, map, rho, step, sign, mom, sb, shares, tab);
    launch_overlapped(true, adj_push_default<real, U>, dim3(nb), 2 * kAdjBlock, 0, s, lat, kcs, map, mom, sb, sign, fbar_prev);
  };
  using T = std::true_type;
  using F = std::false_type;
  if (noise) unit ? pair(T(), T()) : pair(T(), F());
  else unit ? pair(F(), T()) : pair(F(), F());
  return cudaGetLastError();
}

template <class real>
cudaError_t launch_adjoint_gradient_default(const double* shares, const LatticeDev<real>* lat, int n_lat, double* grads,
                                            cudaStream_t s) {
  adj_sum_shares<real><<<dim3(n_lat, 3), 1024, 0, s>>>(shares, lat, grads);
  return cudaGetLastError();
}

#define LB_ADJ_INST(real)                                                                                             \
  template cudaError_t launch_adjoint_step<real>(const real*, const real*, const double*, double*,                    \
                                                 const LatticeDev<real>*, const RowConst<real>*, const AdjConst*,     \
                                                 const AdjMap&, uint32_t, bool, double, bool, double*, double*,       \
                                                 double*, double*, double*, const NormalTables*, cudaStream_t);       \
  template cudaError_t launch_adjoint_densities<real>(const real*, int64_t, int, const LatticeDev<real>*,             \
                                                      const RowConst<real>*, const AdjMap&, double*, float*, int64_t, \
                                                      cudaStream_t);                                                  \
  template cudaError_t launch_adjoint_pressures<real>(const real*, int64_t, int, const LatticeDev<real>*,             \
                                                      const RowConst<real>*, const AdjMap&, const double*,            \
                                                      const float*, int64_t, double*, double*, cudaStream_t);         \
  template cudaError_t launch_adjoint_step_default<real>(const real*, const double*, double*, const LatticeDev<real>*, \
                                                         const AdjConst*, bool, const AdjMap&, uint32_t, bool, double, \
                                                         const double*, double*, double*, double*,                    \
                                                         const NormalTables*, cudaStream_t);                          \
  template cudaError_t launch_adjoint_gradient_default<real>(const double*, const LatticeDev<real>*, int, double*,    \
                                                             cudaStream_t);
LB_ADJ_INST(float)
LB_ADJ_INST(double)

}  // namespace lbk
