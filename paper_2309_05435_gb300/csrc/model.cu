// Theta-dependent model values (Sections 2.1-2.3).
//
// The spatial pattern and the theta-free parts C, G and H = G C^-1 G are
// built once at context creation; here the device turns theta into
//   Q_s = kappa^4 C + 2 kappa^2 G + H            (alpha = 2, lumped mass)
//   dQ_s/dlog kappa = 4 kappa^4 C + 4 kappa^2 G
//   M = (kappa^2 C + G) C^-1/2                    (factor of Q_s = M M^T)
// and the scalars of the unit-variance AR(1) time structure.
#include <algorithm>

#include "kernels.cuh"

namespace qsel {

thread_local int64_t g_launch_count = 0;
thread_local Profiler *g_prof = nullptr;

// Thread per slab, a warp per SM: the binary64 divisions and exponentials are the
// time (one thread for all slabs took 1 us a slab, blocks of eight warps 10 us).
__global__ void __launch_bounds__(32) k_time_coeffs(const double *__restrict__ theta, int n_t, TimeCoeffs tc) {
  const double log_kappa = theta[0], log_tau = theta[1], logit_rho = theta[2];
  const double kappa = exp(log_kappa);
  const double tau = exp(log_tau);
  const double rho = 1.0 / (1.0 + exp(-logit_rho));
  const double om = 1.0 - rho * rho;            // 1 - rho^2
  const double drho_deta = rho * (1.0 - rho);   // d rho / d logit rho
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n_t) {
    // R = B^T B: 1 at both ends, 1 + rho^2 inside (1 - rho^2 for one slab)
    double R, dR;
    if (n_t == 1) {
      R = om;
      dR = -2.0 * rho;
    } else if (t == 0 || t == n_t - 1) {
      R = 1.0;
      dR = 0.0;
    } else {
      R = 1.0 + rho * rho;
      dR = 2.0 * rho;
    }
    tc.a0[t] = tau * R / om;
    tc.r0[t] = tau * drho_deta * (dR / om + R * 2.0 * rho / (om * om));
    tc.bdiag[t] = (t == 0) ? sqrt(om) : 1.0;
    if (t + 1 < n_t) {
      // off-diagonal of R is -rho, of dR/drho is -1
      tc.a1[t] = -tau * rho / om;
      tc.r1[t] = tau * drho_deta * (-1.0 / om - rho * 2.0 * rho / (om * om));
    }
  }
  if (t != 0) return;
  tc.scalars[0] = kappa;
  tc.scalars[1] = tau;
  tc.scalars[2] = rho;
  tc.scalars[3] = sqrt(tau / om);
  tc.scalars[4] = -rho;
}

void launch_time_coeffs(cudaStream_t s, const double *theta_dev, int n_t, TimeCoeffs tc) {
  ++g_launch_count;
  k_time_coeffs<<<(n_t + 31) / 32, 32, 0, s>>>(theta_dev, n_t, tc);
}

__global__ void k_qs_values(int n_ent, const double *__restrict__ c_pat,
                            const double *__restrict__ g_pat, const double *__restrict__ h_pat,
                            const double *__restrict__ isqc_pat, const double *__restrict__ scalars,
                            double *__restrict__ qs, double *__restrict__ dqs,
                            double *__restrict__ kc) {
  const double kappa = scalars[0];
  const double k2 = kappa * kappa;
  const double k4 = k2 * k2;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_ent; e += gridDim.x * blockDim.x) {
    const double c = c_pat[e], g = g_pat[e];
    qs[e] = k4 * c + 2.0 * k2 * g + h_pat[e];
    dqs[e] = 4.0 * k4 * c + 4.0 * k2 * g;
    kc[e] = (k2 * c + g) * isqc_pat[e];
  }
}

void launch_qs_values(cudaStream_t s, int n_ent, const double *c_pat, const double *g_pat,
                      const double *h_pat, const double *isqc_pat, const double *scalars,
                      double *qs, double *dqs, double *kc) {
  ++g_launch_count;
  int grid = (n_ent + 255) / 256;
  if (grid > 1024) grid = 1024;
  if (grid < 1) grid = 1;
  k_qs_values<<<grid, 256, 0, s>>>(n_ent, c_pat, g_pat, h_pat, isqc_pat, scalars, qs, dqs, kc);
}

// ---------------------------------------------------------------------------
// Diffusion-based model (Section 2.2, Eqs. spde:5-8) with (alpha_t, alpha_s,
// alpha_e) = (1, 2, 1): with g = gamma_s^2 and the theta-free pattern arrays
// C, G, H = G C^-1 G, H3 = H C^-1 G,
//   K1 = g C + G,  K2 = g^2 C + 2 g G + H,  K3 = g^3 C + 3 g^2 G + 3 g H + H3,
//   dK_a/dlog gamma_s = 2 g a K_{a-1} (K_0 = C),
// and per slab t with the temporal mass / boundary / stiffness diagonals
// m0, m1, m2 (unit spacing, lumped mass):
//   A_t   = ge2 (m0 K3 + 2 gt m1 K2 + gt^2 m2 K1)               (ge2 = gamma_e^2)
//   dA_s  = ge2 (m0 dK3 + 2 gt m1 dK2 + gt^2 m2 dK1)
//   dA_t  = ge2 (2 gt m1 K2 + 2 gt^2 m2 K1),   dA_e = 2 A_t,
// couplings B_t = -ge2 gt^2 K1 (the stiffness has -1 off the diagonal), with
// dB_s = -ge2 gt^2 dK1, dB_t = 2 B_t, dB_e = 2 B_t.
// Output layout: blk = [A | dA_s | dA_t | dA_e] (n_t x n_ent each), then K1,
// dK1 (n_ent each); coef = [-ge2 gt^2 | -2 ge2 gt^2 | -2 ge2 gt^2] (n_t each).
// ---------------------------------------------------------------------------
__global__ void k_diffusion_values(const double *__restrict__ theta, int n_t, int n_ent,
                                   const double *__restrict__ c_pat, const double *__restrict__ g_pat,
                                   const double *__restrict__ h_pat, const double *__restrict__ h3_pat,
                                   double *__restrict__ blk, double *__restrict__ coef) {
  const double gs = exp(theta[0]), gt = exp(theta[1]), ge = exp(theta[2]);
  const double g = gs * gs, ge2 = ge * ge;
  const int64_t total = (int64_t)n_t * n_ent;
  double *A = blk, *dAs = blk + total, *dAt = blk + 2 * total, *dAe = blk + 3 * total;
  double *K1o = blk + 4 * total, *dK1o = K1o + n_ent;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(q / n_ent);
    const int e = (int)(q - (int64_t)t * n_ent);
    const bool end = (t == 0 || t == n_t - 1);
    const double m0 = (n_t == 1) ? 1.0 : (end ? 0.5 : 1.0);
    const double m1 = (n_t == 1) ? 1.0 : (end ? 0.5 : 0.0);
    const double m2 = (n_t == 1) ? 0.0 : (end ? 1.0 : 2.0);
    const double c = c_pat[e], gg = g_pat[e], h = h_pat[e], h3 = h3_pat[e];
    const double K1 = g * c + gg;
    const double K2 = g * g * c + 2.0 * g * gg + h;
    const double K3 = g * g * g * c + 3.0 * g * g * gg + 3.0 * g * h + h3;
    const double dK1 = 2.0 * g * c, dK2 = 4.0 * g * K1, dK3 = 6.0 * g * K2;
    const double a = ge2 * (m0 * K3 + 2.0 * gt * m1 * K2 + gt * gt * m2 * K1);
    A[q] = a;
    dAs[q] = ge2 * (m0 * dK3 + 2.0 * gt * m1 * dK2 + gt * gt * m2 * dK1);
    dAt[q] = ge2 * (2.0 * gt * m1 * K2 + 2.0 * gt * gt * m2 * K1);
    dAe[q] = 2.0 * a;
    if (t == 0) {
      K1o[e] = K1;
      dK1o[e] = dK1;
    }
    if (e == 0) {
      coef[t] = -ge2 * gt * gt;
      coef[n_t + t] = -2.0 * ge2 * gt * gt;
      coef[2 * n_t + t] = -2.0 * ge2 * gt * gt;
    }
  }
}

void launch_diffusion_values(cudaStream_t s, const double *theta_dev, int n_t, int n_ent, const double *c_pat,
                             const double *g_pat, const double *h_pat, const double *h3_pat, double *blk,
                             double *coef) {
  ++g_launch_count;
  const int64_t total = (int64_t)n_t * n_ent;
  int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 8);
  if (grid < 1) grid = 1;
  k_diffusion_values<<<grid, 256, 0, s>>>(theta_dev, n_t, n_ent, c_pat, g_pat, h_pat, h3_pat, blk, coef);
}

}  // namespace qsel
