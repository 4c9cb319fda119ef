// lb_adjoint.cuh -- host interface of the adjoint sweep (lb_adjoint.cu): the gradient of the
// time-averaged mean-pressure shift with respect to (G, lambda_s, lambda_d).
#pragma once

#include "lb_internal.cuh"

namespace lbk {

// One warp per block: the transposed step takes many registers (128 a thread for the default options,
// bound there, with 16 to 80 bytes spilled; 152 to 184 for the others), so a lattice of a few ten thousand
// sites is fewer threads than the GPU holds, and the smallest blocks spread them most evenly over the SMs
// (measured on 256 x 128 with the kernels of every option: 32 threads 0.476 s per gradient, 128 threads
// 0.504 s).
constexpr int kAdjBlock = 32;
inline int adjoint_blocks(int n_sites) { return (n_sites + kAdjBlock - 1) / kAdjBlock; }

// Per-lattice constants of the transposed step, formed once on the host in double precision from
// the rates and noise amplitudes the device holds.  For sigma^2 = K (2 - lambda) lambda,
// d sigma / d lambda = sigma (1 - lambda) / ((2 - lambda) lambda).
struct AdjConst {
  double oml[9];  // 1 - lambda_a (relaxation, Eq. MRT)
  double ohl[6];  // 1 - lambda_a / 2 (second-order forcing, moments 1..5)
  double dsm;     // d sigma / d lambda_d of the momentum noise (moments 1, 2), hom noise
  double d4, d5;  // d sigma / d lambda_s of moments 4 and 5, hom noise
  // loc noise: sigma_mom = pm sqrt(rho^A rho^B / rho) and sigma^S_a = pa[a] sqrt(rho^S) with the
  // local densities; dpm = d pm / d lambda_d, dp4 and dp5 = d pa[4], pa[5] / d lambda_s
  double pm, dpm, pa[9], dp4, dp5;
  bool options;   // any of no a*, fixed wall composition, loc noise (the kernels that handle them)
  double w_loss;  // 1 / (T N): the loss's weight of one site's pressure at one step (set per call)
  // The default options' kernels: the factors of m^eq (l*), of the source (o*) and of the moments
  // themselves (b*) with 1/N_a and the weights of the links folded in (adj_local_default).
  double l1, l3, l4, o1, o3, o4, o5, b1, b3, b4, b6, b8;
  bool unit;      // the rates of moments 3..8 are 1: their b* vanish
};

template <class real>
inline AdjConst adjoint_constants(const LatticeDev<real>& L) {
  AdjConst k;
  for (int a = 0; a < 9; ++a) k.oml[a] = 1 - (double)L.lam[a];
  for (int a = 0; a < 6; ++a) k.ohl[a] = 1 - 0.5 * (double)L.lam[a];
  auto dsigma = [](double sigma, double lam) { return sigma * (1 - lam) / ((2 - lam) * lam); };
  const double ld = (double)L.lam[1], ls = (double)L.lam[4];
  k.dsm = dsigma((double)L.sig_mom, ld);
  k.d4 = dsigma((double)L.sig[4], ls);
  k.d5 = dsigma((double)L.sig[5], ls);
  k.pm = (double)L.pref_mom;
  k.dpm = dsigma(k.pm, ld);
  for (int a = 0; a < 9; ++a) k.pa[a] = a >= 3 ? (double)L.pref[a] : 0.0;
  k.dp4 = dsigma(k.pa[4], ls);
  k.dp5 = dsigma(k.pa[5], ls);
  const double le = (double)L.lam[3], lq = (double)L.lam[6], leps = (double)L.lam[8];
  k.l1 = ld / 12, k.l3 = le / 12, k.l4 = ls / 4;
  k.o1 = (1 - 0.5 * ld) / 12, k.o3 = (1 - 0.5 * le) / 6, k.o4 = (1 - 0.5 * ls) / 2, k.o5 = (1 - 0.5 * ls) / 4;
  k.b1 = (1 - ld) / 12, k.b3 = (1 - le) / 36, k.b4 = (1 - ls) / 4, k.b6 = (1 - lq) / 12, k.b8 = (1 - leps) / 72;
  k.unit = L.flags & DF_UNIT;
  k.options = !(L.flags & DF_ASTAR) || (L.flags & (DF_WALL_FIXED | DF_NOISE_LOC));
  return k;
}

// The adjoint's blocks over a batch: the blocks of lattice i are first[i] .. first[i + 1] - 1
// (adjoint_blocks of its sites each), lat_of[b] the lattice of block b; so every block belongs to
// one lattice and a lattice's blocks and sums are those of the lattice alone.  Device arrays.
struct AdjMap {
  const int* lat_of;  // [n_blocks]
  const int* first;   // [n_lat + 1]
  int n_blocks, n_lat;
};

// One adjoint step of every lattice of the batch: from fbar (sensitivity to f*_k) and the forward
// state f_prev = f*_{k-1}, write fbar_prev and add this step's gradient share, block by block, to
// partials (3 doubles per block, zeroed before the sweep); then launch_adjoint_gradient sums each
// lattice's blocks into grads[3 i ..].  The site-indexed buffers hold the lattices one after
// another at their site offsets (LatticeDev::site_off): rho 2, fl and fbar 18, sb 4 doubles per
// site; the states have the context's layout (LatticeDev::f_off).  rho holds the densities of
// f_prev if rho_ready, else they are computed first; with f_next = f*_{k-2} given, its densities
// go to rho_next for the next step.  kcs: the lattices' AdjConst (device); options: any lattice
// uses a non-default option of the step; sign: +1 for the noisy run, -1 for the noiseless one
// (the loss weight of a site is sign w_loss).  The sensitivities are double precision for either
// state precision.
template <class real>
cudaError_t launch_adjoint_step(const real* f_prev, const real* f_next, const double* fbar, double* fbar_prev,
                                const LatticeDev<real>* lat, const RowConst<real>* rows, const AdjConst* kcs,
                                const AdjMap& map, uint32_t step, bool noise, double sign, bool rho_ready, double* rho,
                                double* rho_next, double* fl, double* sb, double* partials, const NormalTables* tab,
                                cudaStream_t s);
cudaError_t launch_adjoint_gradient(const double* partials, const AdjMap& map, double* grads, cudaStream_t s);

// The same for lattices of the default options (AdjConst::options false for all), whose densities and
// pressures come for all states of a segment at once.  n_states states at f, f + S, ..; NS: sites of the
// batch.  rho: [2][N] per lattice at 2 site_off, 2 NS doubles per state (FP32 states may pass null); dev:
// FP32 states only, the density deviations as the step kernels sum them, 2 NS floats per state.
template <class real>
cudaError_t launch_adjoint_densities(const real* f, int64_t S, int n_states, const LatticeDev<real>* lat,
                                     const RowConst<real>* rows, const AdjMap& map, double* rho, float* dev, int64_t NS,
                                     cudaStream_t s);
// out[state * n_lat + lattice]: the pressure summed over the lattice's sites (minus the background in
// FP32); part: n_blocks doubles per state.
template <class real>
cudaError_t launch_adjoint_pressures(const real* f, int64_t S, int n_states, const LatticeDev<real>* lat,
                                     const RowConst<real>* rows, const AdjMap& map, const double* rho, const float* dev,
                                     int64_t NS, double* part, double* out, cudaStream_t s);
// Buffers per site: mom up to 18 doubles, sb 8, shares 3 ([3][N] per lattice at 3 site_off, zeroed before
// the sweep).  rho: the densities of f_prev.  unit: every lattice's rates of moments 3..8 are 1.
template <class real>
cudaError_t launch_adjoint_step_default(const real* f_prev, const double* fbar, double* fbar_prev,
                                        const LatticeDev<real>* lat, const AdjConst* kcs, bool unit, const AdjMap& map,
                                        uint32_t step, bool noise, double sign, const double* rho, double* mom, double* sb,
                                        double* shares, const NormalTables* tab, cudaStream_t s);
template <class real>
cudaError_t launch_adjoint_gradient_default(const double* shares, const LatticeDev<real>* lat, int n_lat, double* grads,
                                            cudaStream_t s);

}  // namespace lbk
