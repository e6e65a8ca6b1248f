// pe_prep.cuh -- row A1: per-sample coefficients from theta[11], and their derivatives for the gradient, with G threads
// to a sample (arXiv:2602.12011 Sec. 2.1-2.3).
//  TaylorF2 phase (Buonanno et al. 2009 3.5PN; 1.5PN spin-orbit, 2PN aligned spin-spin),
//  SPA amplitudes of the leading-order spherical modes (Blanchet 2014), C-infinity taper
//  on the orbital frequency between 0.9 F_isco and F_isco, -2Y_lm polarisation weights
//  (h_{l,-m} = (-1)^l h*_lm), sky frame.
//
// What bounds it: one thread's chain of ~1,500 FP64 instructions (five sincos, a cube root, a log, square roots and
// divisions, five modes) at ~50 cycles each, 38 us whatever the batch, half of a single-sample call. The pieces are
// independent, so eight threads of a warp share a sample: its sines and cosines, modes and converted coefficients
// are then one instruction stream each. From kPrepSerialB samples on one thread per sample issues fewer instructions in
// all (whole calls on a grid of four bins, eight threads against one: 4,096 samples 112 and 121 us, gradients 311 and 324; 6,144: 165 and 162,
// gradients 435 and 426; 8,192: 186 and 173; 65,536: 1144 and 858). Both run the same pieces (not inlined, exchanged through memory), so a
// sample's coefficients are the same bits in any batch.
#pragma once
#include "pe_device.cuh"

namespace pe {

constexpr int kPrepThreads = 64;
constexpr int kPrepGroup = 8;
constexpr int kPrepSerialB = 6144;

// Values shared by the pieces of one sample.
struct PrepTmp {
  double sc[5][2];   // sin, cos of lambda, beta, psi, iota, iota/2
  double M, eta, m1, m2, delta, n, Fisco;
  double cm1, lncm1;
  double P[8], Q5, Q6;
  double amp[kNModes], ph0[kNModes], fend[kNModes];
  int active[kNModes];
};

// piece i of the first stage: 0..4 the angles, 5 the mass ratios, 6 the chirp scale
static __device__ __noinline__ void prep_base(const double* th, int i, PrepTmp& t) {
  if (i < 5) {
    const double x = i == 0 ? th[7] : (i == 1 ? th[8] : (i == 2 ? th[9] : (i == 3 ? th[5] : 0.5 * th[5])));
    sincos(x, &t.sc[i][0], &t.sc[i][1]);
  } else if (i == 5) {
    const double q = th[1], iq = 1.0 / (1.0 + q);
    t.eta = q / ((1.0 + q) * (1.0 + q));
    t.m1 = q * iq;
    t.m2 = iq;
    t.delta = (q - 1.0) * iq;
    t.n = 3.0 / (128.0 * t.eta);
  } else if (i == 6) {
    const double M = th[0] * kMsunS;
    t.M = M;
    t.Fisco = 1.0 / (k6Pow15 * 2.0 * kPi * M);
    t.cm1 = cbrt(2.0 * kPi * M);
    t.lncm1 = log(2.0 * kPi * M) * (1.0 / 3.0);
  }
}

// the PN series (before its derivatives in v) and the sky frame
static __device__ __noinline__ void prep_series(const double* th, PrepTmp& t) {
  const double pi = kPi, chi1 = th[2], chi2 = th[3], eta = t.eta, n = t.n;
  const double bso = chi1 * (113.0 / 12.0 * t.m1 * t.m1 + 25.0 / 4.0 * eta) + chi2 * (113.0 / 12.0 * t.m2 * t.m2 + 25.0 / 4.0 * eta);
  const double sss = 79.0 / 8.0 * eta * chi1 * chi2;
  const double a5c = pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta);
  const double a6c = 11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * pi * pi - 6848.0 / 21.0 * kEulerGamma +
                     (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi * pi) * eta + 76055.0 / 1728.0 * eta * eta -
                     127825.0 / 1296.0 * eta * eta * eta;
  t.P[0] = n;
  t.P[1] = 0.0;
  t.P[2] = n * (3715.0 / 756.0 + 55.0 / 9.0 * eta);
  t.P[3] = n * (-16.0 * pi + 4.0 * bso);
  t.P[4] = n * (15293365.0 / 508032.0 + 27145.0 / 504.0 * eta + 3085.0 / 72.0 * eta * eta - 10.0 * sss);
  t.P[5] = n * a5c * (1.0 + 1.5 * kLn6);                // alpha5 (1 + 3 ln(v/v_lso)), v_lso = 6^-1/2
  t.P[6] = n * (a6c - 6848.0 / 21.0 * kLn4);            // alpha6 - (6848/21) ln(4 v)
  t.P[7] = n * pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta * eta);
  t.Q5 = n * 3.0 * a5c;
  t.Q6 = n * (-6848.0 / 21.0);
}
static __device__ __noinline__ void prep_frame(const double* th, const PrepTmp& t, SampleCoef& S) {
  const double sl = t.sc[0][0], cl = t.sc[0][1], sb = t.sc[1][0], cb = t.sc[1][1], sp = t.sc[2][0], cp = t.sc[2][1];
  const double k[3] = {-(cb * cl), -(cb * sl), -sb}, u[3] = {sl, -cl, 0.0}, v[3] = {-(sb * cl), -(sb * sl), cb};
  for (int i = 0; i < 3; ++i) {
    S.k[i] = k[i];
    S.p[i] = cp * u[i] + sp * v[i];
    S.q[i] = -(sp * u[i]) + cp * v[i];
    S.kw[i] = to_dw(k[i]);
  }
  S.tc = th[10];
  S.tcw = to_dw(th[10]);
}

// mode md's coefficients that need nothing of the other modes
static __device__ __noinline__ void prep_mode(const double* th, int md, bool valid, unsigned mask, PrepTmp& t, SampleCoef& S) {
  ModeCoef& C = S.md[md];
  const int l = kModeL[md], m = kModeM[md];
  const int p = md == 0 ? 0 : (md < 3 ? 1 : 2);
  // |H_lm| / x^(p/2) and arg(conj H_lm) in turns
  const double odd = md == 1 ? 1.0 / 3.0 : 0.75 * 1.0350983390135313;                            // 3/4 sqrt(15/14)
  const double even = (md == 3 ? 1.0 / 3.0 : 8.0 / 9.0) * 0.84515425472851658;                  // sqrt(5/7)
  const double hmag = md == 0 ? 1.0 : (p == 1 ? odd * t.delta : even * (1.0 - 3.0 * t.eta));
  const double argt = md == 1 ? -0.25 : (md == 2 ? 0.25 : (md == 4 ? 0.5 : 0.0));
  const double cm = t.cm1 * kCbrtInv[m], icm = 1.0 / cm;
  C.cm = cm;
  C.icm = icm;
  C.lncm = t.lncm1 - kLnM3[m];
  const double D = th[4] * kGpcS;
  C.amp = 2.0 * kPi * t.M * t.M / D * sqrt(t.eta / (3.0 * m)) * hmag * (icm * icm * icm * rsqrt(cm));
  const double icm2 = icm * icm;
  C.icm5 = icm2 * icm2 * icm;
  C.ampp = p == 0 ? C.amp : (p == 1 ? C.amp * cm : C.amp * cm * cm);
  const double ph = m * (th[6] * (0.5 / kPi)) + (0.125 + argt);
  C.ph0 = ph - rint(ph);
  C.mfac = m * (0.25 / kPi);
  C.tffac = m * (1.0 / (12.0 * kPi));
  double yp, yn;
  sylm_pair(l, m, t.sc[3][1], t.sc[3][0], t.sc[4][1], t.sc[4][0], &yp, &yn);
  const double sgn = (l % 2) ? -1.0 : 1.0;
  C.Pp = 0.5 * (yp + sgn * yn);
  C.Pc = 0.5 * (sgn * yn - yp);
  C.Pc2 = sgn * yn - yp;
  C.fend = m * t.Fisco;
  C.ftap = 0.9 * m * t.Fisco;
  C.Ppw = to_dw(C.Pp);
  C.Pcw = to_dw(C.Pc);
  C.cmw = to_dw(cm);
  C.tffacw = to_dw(C.tffac);
  C.ph0w = to_dw(C.ph0);
  C.p = p;
  C.active = (valid && (mask & (1u << md)) && hmag != 0.0) ? 1 : 0;
  t.amp[md] = C.amp;
  t.ph0[md] = C.ph0;
  t.fend[md] = C.fend;
  t.active[md] = C.active;
}

// piece i of the last stage: 0..7 the series' derivatives and double words, 8 what joins the modes, 9..13 mode
// i - 9's amplitude as a double word, 14 the logarithmic terms
static __device__ __noinline__ void prep_rest(int i, bool valid, const PrepTmp& t, SampleCoef& S) {
  const double a0 = t.amp[0];
  const int e0 = (a0 > 0.0 && isfinite(a0)) ? ilogb(a0) : 0;
  if (i < 8) {
    const double P = t.P[i], Pd = double(i - 5) * P;
    S.P[i] = P;
    S.Pd[i] = Pd;
    S.Pdd[i] = double(i - 5) * Pd;
    S.Pw[i] = to_dw(P);
    S.Pdw[i] = to_dw(Pd);
  } else if (i == 8) {
    S.valid = valid ? 1 : 0;
    S.hsc = scalbn(1.0, -e0);
    S.ihsc = scalbn(1.0, e0);
    S.pair32 = (t.active[0] && t.active[3]) ? 1 : 0;
    double2 k32 = make_double2(0.0, 0.0);
    if (S.pair32) {
      double sd, cd;
      sincospi(2.0 * (t.ph0[3] - t.ph0[0]), &sd, &cd);
      const double r = t.amp[3] / a0;
      k32 = make_double2(r * cd, r * sd);
    }
    S.k32 = k32;
    S.k32w[0] = to_dw(k32.x);
    S.k32w[1] = to_dw(k32.y);
  } else if (i < 14) {
    S.md[i - 9].ampw = to_dw(t.amp[i - 9] * scalbn(1.0, -e0));
  } else {
    S.Q5 = t.Q5;
    S.Q6 = t.Q6;
    S.Q5w = to_dw(t.Q5);
    S.Q6w = to_dw(t.Q6);
  }
}

// Derivatives of the coefficients the adjoint needs (SampleGrad), in closed form: piece 0 the series in q, chi1 and
// chi2, piece 1 the sky frame, pieces 2..6 mode i - 2.
static __device__ __noinline__ void prep_grad_piece(const double* th, int i, const PrepTmp& t, const SampleCoef& S, SampleGrad& G) {
  const double pi = kPi, q = th[1], eta = t.eta, n = t.n;
  const double m2 = t.m2, dm1 = m2 * m2;                     // d m1/dq = 1/(1+q)^2 = -d m2/dq
  const double deta = (1.0 - q) * m2 * m2 * m2;              // d eta/dq
  if (i == 0) {
    const double dn = -deta / eta;                           // d ln n/dq
    const double m1 = t.m1, c1 = th[2], c2 = th[3];
    const double dbso = c1 * (113.0 / 6.0 * m1 * dm1 + 25.0 / 4.0 * deta) + c2 * (-113.0 / 6.0 * m2 * dm1 + 25.0 / 4.0 * deta);
    const double da5 = pi * (-65.0 / 9.0) * deta;
    double d[8];
    d[0] = 0.0;
    d[1] = 0.0;
    d[2] = 55.0 / 9.0 * deta;
    d[3] = 4.0 * dbso;
    d[4] = deta * (27145.0 / 504.0 + 3085.0 / 36.0 * eta - 790.0 / 8.0 * c1 * c2);
    d[5] = da5 * (1.0 + 1.5 * kLn6);
    d[6] = deta * ((-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi * pi) + 76055.0 / 864.0 * eta - 127825.0 / 432.0 * eta * eta);
    d[7] = pi * deta * (378515.0 / 1512.0 - 74045.0 / 378.0 * eta);
    for (int k = 0; k < 8; ++k) {
      const double dP = n * d[k] + t.P[k] * dn;
      G.dP_dq[k] = dP;
      G.dPd_dq[k] = double(k - 5) * dP;
    }
    G.dQ5_dq = n * 3.0 * da5 + t.Q5 * dn;
    G.dQ6_dq = t.Q6 * dn;
    G.dP3_dc1 = n * 4.0 * (113.0 / 12.0 * m1 * m1 + 25.0 / 4.0 * eta);
    G.dP3_dc2 = n * 4.0 * (113.0 / 12.0 * m2 * m2 + 25.0 / 4.0 * eta);
    G.dP4_dc1 = n * (-790.0 / 8.0) * eta * c2;
    G.dP4_dc2 = n * (-790.0 / 8.0) * eta * c1;
    G.dlnA_ddL = -1.0 / th[4];
  } else if (i == 1) {
    const double sl = t.sc[0][0], cl = t.sc[0][1], sb = t.sc[1][0], cb = t.sc[1][1], sp = t.sc[2][0], cp = t.sc[2][1];
    // u = (sl, -cl, 0), v = (-sb cl, -sb sl, cb); k = -(cb cl, cb sl, sb)
    const double u[3] = {sl, -cl, 0.0}, v[3] = {-(sb * cl), -(sb * sl), cb};
    const double ul[3] = {cl, sl, 0.0}, vl[3] = {sb * sl, -(sb * cl), 0.0}, vb[3] = {-(cb * cl), -(cb * sl), -sb};
    const double kl[3] = {cb * sl, -(cb * cl), 0.0}, kb[3] = {sb * cl, sb * sl, -cb};
    for (int c = 0; c < 3; ++c) {
      G.dk[c][0] = kl[c];
      G.dk[c][1] = kb[c];
      G.dk[c][2] = 0.0;
      G.dp[c][0] = cp * ul[c] + sp * vl[c];
      G.dp[c][1] = sp * vb[c];
      G.dp[c][2] = cp * v[c] - sp * u[c];
      G.dq[c][0] = cp * vl[c] - sp * ul[c];
      G.dq[c][1] = cp * vb[c];
      G.dq[c][2] = -(cp * u[c]) - sp * v[c];
    }
  } else {
    const int md = i - 2, l = kModeL[md];
    ModeGrad& M = G.md[md];
    const bool some = t.amp[md] != 0.0;
    // amp ~ M^2 cm^(-7/2) sqrt(eta) hmag, cm ~ M^(1/3); hmag ~ 1, delta or 1 - 3 eta
    const double dh = md == 0 ? 0.0 : (md < 3 ? 2.0 * dm1 / t.delta : -3.0 * deta / (1.0 - 3.0 * eta));
    M.dlnA_dM = some ? (5.0 / 6.0) / th[0] : 0.0;
    M.dlnA_dq = some ? 0.5 * deta / eta + dh : 0.0;
    M.dcm_dM = S.md[md].cm / (3.0 * th[0]);
    M.dfend_dM = -t.fend[md] / th[0];
    const double si = t.sc[3][0], ci = t.sc[3][1], s = t.sc[4][0], c = t.sc[4][1];
    double yp, yn;   // d/d iota of sylm_pair
    if (md == 0) {
      const double K = sqrt(5.0 / (64.0 * pi));
      yp = -2.0 * K * (1.0 + ci) * si;
      yn = 2.0 * K * (1.0 - ci) * si;
    } else if (md == 1) {
      const double K = sqrt(5.0 / (16.0 * pi));
      yp = K * (ci * (1.0 + ci) - si * si);
      yn = K * (ci * (1.0 - ci) + si * si);
    } else if (md == 2) {
      const double K = 0.5 * sqrt(21.0 / (2.0 * pi)), c4 = c * c * c * c, s4 = s * s * s * s;
      yp = -K * c4 * (c * c - 5.0 * s * s);
      yn = K * s4 * (5.0 * c * c - s * s);
    } else if (md == 3) {
      const double K = 0.5 * sqrt(7.0 / pi), K2 = sqrt(7.0 / (4.0 * pi)), c4 = c * c * c * c, s4 = s * s * s * s;
      yp = -K * (2.0 * c * c * c * s * (3.0 * ci - 2.0) + 3.0 * c4 * si);
      yn = K2 * (2.0 * s * s * s * c * (3.0 * ci + 2.0) - 3.0 * s4 * si);
    } else {
      const double K = 3.0 * sqrt(7.0 / pi), c2 = c * c, s2 = s * s;
      yp = K * c2 * c2 * c * s * (c2 - 3.0 * s2);
      yn = K * s2 * s2 * s * c * (3.0 * c2 - s2);
    }
    const double sgn = (l % 2) ? -1.0 : 1.0;
    M.dPp_di = 0.5 * (yp + sgn * yn);
    M.dPc_di = 0.5 * (sgn * yn - yp);
  }
}

// Active bins of a detector: the bins below the largest active mode's taper end (one extra bin guards the rounding of
// the bound; every unit still checks f < fend of its own mode).
__device__ __forceinline__ int active_bins(const DetDev& D, double fmax) {
  if (!(fmax > 0.0)) return 0;
  const double kx = ceil(fmax * D.T) - double(D.k0) + 1.0;
  return kx <= 0.0 ? 0 : (kx >= double(D.nb) ? D.nb : int(kx));
}

// One sample's coefficients by G threads of a warp (lane: the thread's place in the group).
template <int G, bool GRAD>
__device__ __forceinline__ void prep_sample(const double* th, unsigned mask, const DetSet& ds, int B, int s, int lane, PrepTmp& t,
                                            SampleCoef& S, SampleGrad* grad, int* nend, int* status) {
  const bool valid = theta_valid(th);
  const unsigned group = G == 1 ? 0u : ((1u << G) - 1u) << ((threadIdx.x & 31) / G * G);
#pragma unroll 1
  for (int i = lane; i < 7; i += G) prep_base(th, i, t);
  if (G > 1) __syncwarp(group);
#pragma unroll 1
  for (int i = lane; i < 7; i += G) {
    if (i < kNModes) prep_mode(th, i, valid, mask, t, S);
    else if (i == 5) prep_series(th, t);
    else prep_frame(th, t, S);
  }
  if (G > 1) __syncwarp(group);
#pragma unroll 1
  for (int i = lane; i < 15; i += G) prep_rest(i, valid, t, S);
  if (GRAD) {
#pragma unroll 1
    for (int i = lane; i < 7; i += G) prep_grad_piece(th, i, t, S, *grad);
  }
  double fmax = 0.0;
#pragma unroll
  for (int md = 0; md < kNModes; ++md)
    if (t.active[md]) fmax = fmax > t.fend[md] ? fmax : t.fend[md];
#pragma unroll 1
  for (int I = lane; I < ds.ndet; I += G) nend[I * B + s] = active_bins(ds.d[I], fmax);
  if (status && lane == 0) status[s] = valid ? 0 : 1;
}

template <int G, bool GRAD>
__global__ void __launch_bounds__(kPrepThreads) k_prep(const double* theta, int B, unsigned mask, DetSet ds, SampleCoef* coef,
                                                       SampleGrad* grad, int* nend, int* status) {
  __shared__ PrepTmp tmp[kPrepThreads / G];
  const int g = threadIdx.x / G, s = blockIdx.x * (kPrepThreads / G) + g;
  if (s < B)
    prep_sample<G, GRAD>(theta + (size_t)s * PE_NPARAM, mask, ds, B, s, threadIdx.x % G, tmp[g], coef[s],
                         GRAD ? grad + s : nullptr, nend, status);
}

template <bool GRAD>
cudaError_t prep_launch(const double* theta, int B, unsigned mask, const DetSet& ds, SampleCoef* coef, SampleGrad* grad,
                        int* nend, int* status, cudaStream_t st) {
  if (B < kPrepSerialB) {
    constexpr int per = kPrepThreads / kPrepGroup;
    k_prep<kPrepGroup, GRAD><<<(B + per - 1) / per, kPrepThreads, 0, st>>>(theta, B, mask, ds, coef, grad, nend, status);
  } else {
    k_prep<1, GRAD><<<(B + kPrepThreads - 1) / kPrepThreads, kPrepThreads, 0, st>>>(theta, B, mask, ds, coef, grad, nend, status);
  }
  return launch_status();
}

}  // namespace pe
