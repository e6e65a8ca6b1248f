// pe_adjoint_fx.cuh -- reverse sweep of the fixed-point unit (pe_device_fx.cuh) for the gradient (row G1) and the Fisher
// matrix (row G2); arXiv:2602.12011 Sec. 2.1-2.3. The forward pass writes each unit's tape (kFt* fields); given the
// bin's link seeds (link_seeds, pe_adjoint_tape.cuh, as integers with one exponent per bin), the sweep pulls them back through
// the link factors, polarisation weights, sincs, norms and phases in fixed point, and only the scalars it ends in (the
// phase's, amplitude's, t_f's and weights' cotangents) return to FP64 for the PN chain rule.
//
// What bounds it: the FP64 forward and reverse it replaces issued 619 FP64 instructions per unit at 1.67 per SM and clock; here
// 141 are left, 34 of them the forward's, most of the others the PN series' derivatives in v and q.
//
// The sky frame enters through rotations: a change of (lambda, beta, psi) turns (k, p, q) rigidly, dk = w x k and so on,
// so the frame's cotangent is three numbers, W.w = sum over links of (projections' cotangents) x (projections), summed per
// bin in place of 42 sums per tile over the tape.
//
// Scales: seeds are below 1/16 at exponent Es (value = n 2^(Es - 1078)), amplitudes below 1/8 (n 2^(E - 1079)); then every
// sum of products here stays inside the formats (|cotangent of a projection| < 0.4, sums of three below 1.2).
#pragma once
#include "pe_adjoint_tape.cuh"
#include "pe_device_fx.cuh"

namespace pe {

// The tape of one thread: field f at p[f * kTileBins] of the CTA's region in global memory, held in L2 by the evict-last
// hint (tape_l2_policy).
struct FxTape {
  static constexpr bool kOn = true, kChain = false;
  double* p;
  unsigned long long pol;
  __device__ __forceinline__ void st(int f, fx v) const { tst(p + f * kTileBins, __longlong_as_double(v), pol); }
  __device__ __forceinline__ fx ld(int f) const { return __double_as_longlong(tld(p + f * kTileBins, pol)); }
};
static_assert((int)kFtFields <= (int)kTapeF, "the regions are those of the FP64 tape");

// The seeds' common factors of one unit's chain rule (doubles): the weights times the amplitude, then v dPsi/dv, v dD/dv, dPsi/dq, dD/dq,
// 1/v, cos and sin of the centre's angle and d(ln taper)/d Mtot. One sweep per unit forms them in place; the Fisher
// matrix's six sweeps read them from the tape (kFtChain on).
struct FxChain {
  double dv, ddv, pq, dq, iv, co, so, tap;
};
enum : int { kFtChain = kFtFields, kFtWeights = kFtChain + 8, kFtAll = kFtWeights + 4 };
__device__ __forceinline__ void fx_weights(const SampleCoef& S, const ModeCoef& C, const ModeCoef* C2, double amp, double v, double2& Ap,
                                           double2& Ac) {
  Ap = make_double2(amp * C.Pp, 0.0);
  Ac = make_double2(amp * C.Pc2, 0.0);
  if (C2) {
    const double2 kap = make_double2(S.k32.x * (v * v), S.k32.y * (v * v));
    Ap = make_double2(amp * fma(kap.x, C2->Pp, C.Pp), amp * (kap.y * C2->Pp));
    Ac = make_double2(amp * fma(kap.x, C2->Pc2, C.Pc2), amp * (kap.y * C2->Pc2));
  }
}
__device__ __forceinline__ FxChain fx_chain(const DetDev& D, const SampleCoef& S, const SampleGrad& SG, const ModeCoef& C,
                                            const ModeGrad& CG, const FxBin& B, double fm13, double v, double w, fx cq, fx sq) {
  FxChain h;
  const double lnv = C.lncm + B.lnf3, iv5 = C.icm5 * D.fm53[B.b];
  // Psi_PN(v), D(v): v dPsi/dv = D, v dD/dv = v^-5 ddpol + Q6 v (2 + ln v); v ~ M^(1/3)
  double dpol = S.Pd[7], ddpol = S.Pdd[7], pq = SG.dP_dq[7], dq = SG.dPd_dq[7];
#pragma unroll
  for (int k = 6; k >= 0; --k) {
    dpol = fma(dpol, v, S.Pd[k]);
    ddpol = fma(ddpol, v, S.Pdd[k]);
    pq = fma(pq, v, SG.dP_dq[k]);
    dq = fma(dq, v, SG.dPd_dq[k]);
  }
  const double q6v = S.Q6 * v, dq6v = SG.dQ6_dq * v;
  h.dv = fma(iv5, dpol, fma(q6v, 1.0 + lnv, S.Q5));
  h.ddv = fma(iv5, ddpol, q6v * (2.0 + lnv));
  h.pq = fma(iv5, pq, lnv * (dq6v + SG.dQ5_dq));
  h.dq = fma(iv5, dq, fma(dq6v, 1.0 + lnv, SG.dQ5_dq));
  h.iv = C.icm * fm13;
  h.co = fx_to_double(cq, -60);
  h.so = fx_to_double(sq, -60);
  h.tap = 0.0;
  if (dlt_pos(C.ftap, B.f)) {
    const double fe = C.fend, ft = C.ftap, A = fe - ft;
    const double dz = 0.1 / (fe - B.f) - A / ((fe - B.f) * (fe - B.f)) - 0.1 / (B.f - ft) -
                      0.9 * A / ((B.f - ft) * (B.f - ft));
    h.tap = -(1.0 - w) * dz * CG.dfend_dM;
  }
  return h;
}

// Scalars of one unit's sweep, in FP64.
struct FxBwd {
  double th;        // cotangent of the phase (rad), summed over the links' angles
  double lnA;       // of ln amplitude
  double alpha, geo;   // of the centre's angle and the constellation's (rad), without the Doppler term
  double W[3];      // of the frame's rotation about k, p, q, without the Doppler term
  double2 Ap, Ac;   // of the weights times the amplitude
};

// seeds: the bin's P_l, Q_l (x, y each) at seeds[(4 l + i) * SST]; Ap, Ac the weights times the amplitude.
template <int SST, class Tape>
__device__ __forceinline__ void fx_bwd(const FxBin& B, fx a3, const volatile fx* seeds, int Es, double2 Ap, double2 Ac, bool pair,
                                       bool helio, const fx* __restrict__ pc, const Tape& tape, FxBwd& o) {
  int E = max(fx_expo(Ap.x), fx_expo(Ac.x));
  if (pair) E = max(E, max(fx_expo(Ap.y), fx_expo(Ac.y)));
  const int ash = 1079 - E;
  fxs Apx = {0, 0}, Acx = {0, 0}, Apy = {0, 0}, Acy = {0, 0};
  const bool some = E >= kFxLeastE;
  if (some) {   // else the weights vanish, and only their own cotangents are not zero
    Apx = fx_split(fx_from_bits(Ap.x, ash));
    Acx = fx_split(fx_from_bits(Ac.x, ash));
  }
  if (pair && some) {
    Apy = fx_split(fx_from_bits(Ap.y, ash));
    Acy = fx_split(fx_from_bits(Ac.y, ash));
  }
  const fxs a4s = fx_split(B.a4), a3s = fx_split(a3);
  fx th0 = 0, th1 = 0, th2 = 0, lnA = 0, Wk = 0, Wp = 0, Wq = 0;
  fx Apb[2] = {0, 0}, Acb[2] = {0, 0}, obb[4] = {0, 0, 0, 0};
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    const int tl = kFtL + kFtLink * l;
    const fxs Px = fx_split(seeds[(4 * l) * SST]), Py = fx_split(seeds[(4 * l + 1) * SST]);
    const fxs Qx = fx_split(seeds[(4 * l + 2) * SST]), Qy = fx_split(seeds[(4 * l + 3) * SST]);
    const fxs kr = fx_split(tape.ld(tl + kFtK)), pr = fx_split(tape.ld(tl + kFtP)), qr = fx_split(tape.ld(tl + kFtQ));
    const fxs inv = fx_split(tape.ld(tl + kFtInv));
    const fxs ec = fx_split(tape.ld(tl + kFtEc)), es = fx_split(tape.ld(tl + kFtEs));
    const fxs sp = fx_split(tape.ld(tl + kFtSp)), sm = fx_split(tape.ld(tl + kFtSm));
    const fxs kn = fx_split(fx_mul(kr, inv));
    const fx npq = fx_mul(pr, inv), nqq = fx_mul(qr, inv);
    const fxs np = fx_split(npq), nq = fx_split(nqq);
    const fxs Fp = fx_split(fx_mul(fx_split(npq - nqq), fx_split(npq + nqq))), Fc = fx_split(fx_mul(np, nq));
    // gam = Fp Ap + i Fc Ac, G = gam E
    fxs gx, gy;
    if (pair) {
      gx = fx_split(fx_msub(Apx, Fp, Acy, Fc));
      fxa g = fx_prod<2>(Apy, Fp);
      fx_mac(g, Acx, Fc);
      gy = fx_split(fx_val(g));
    } else {
      gx = fx_split(fx_mul(Apx, Fp));
      gy = fx_split(fx_mul(Acx, Fc));
    }
    const fxs Gx = fx_split(fx_msub(gx, ec, gy, es));
    fxa t = fx_prod<2>(gx, es);
    fx_mac(t, gy, ec);
    const fxs Gy = fx_split(fx_val(t));
    // Gb = s- P + s+ Q; cotangents of s-+ are Re(G conj P), Re(G conj Q)
    t = fx_prod<2>(sm, Px);
    fx_mac(t, sp, Qx);
    const fxs Gbx = fx_split(fx_val(t));
    t = fx_prod<2>(sm, Py);
    fx_mac(t, sp, Qy);
    const fxs Gby = fx_split(fx_val(t));
    t = fx_prod<2>(Gx, Px);
    fx_mac(t, Gy, Py);
    const fxs smb = fx_split(fx_val(t));
    t = fx_prod<2>(Gx, Qx);
    fx_mac(t, Gy, Qy);
    const fxs spb = fx_split(fx_val(t));
    // d s-+/d kn = -+ a sinc'(u-+)
    const fxs dp = fx_split(tape.ld(tl + kFtDp)), dm = fx_split(tape.ld(tl + kFtDm));
    const fxs knb = fx_split(fx_mul(fx_split(fx_msub(spb, dp, smb, dm)), a4s) << 2);
    // gamb = Gb conj E; the angle's cotangent Im(Gb conj G)
    t = fx_prod<2>(Gbx, ec);
    fx_mac(t, Gby, es);
    const fx gbxq = fx_val(t);
    const fx gbyq = fx_msub(Gby, ec, Gbx, es);
    const fxs gbx = fx_split(gbxq), gby = fx_split(gbyq);
    const fx th = fx_msub(Gby, Gx, Gbx, Gy);
    if (l == 0) th0 = th;
    else if (l == 1) th1 = th;
    else th2 = th;
    t = fx_prod<2>(gbx, gx);
    fx_mac(t, gby, gy);
    lnA += fx_val(t);
    Apb[0] += fx_mul(gbx, Fp);
    Acb[0] += fx_mul(gby, Fc);
    fxs Fpb, Fcb;
    if (pair) {
      Apb[1] += fx_mul(gby, Fp);
      Acb[1] -= fx_mul(gbx, Fc);
      t = fx_prod<2>(gbx, Apx);
      fx_mac(t, gby, Apy);
      Fpb = fx_split(fx_val(t));
      Fcb = fx_split(fx_msub(gby, Acx, gbx, Acy));
    } else {
      Fpb = fx_split(fx_mul(gbx, Apx));
      Fcb = fx_split(fx_mul(gby, Acx));
    }
    // Fp = np^2 - nq^2, Fc = np nq
    const fxs npb = fx_split(2 * fx_mul(np, Fpb) + fx_mul(nq, Fcb));
    const fxs nqb = fx_split(fx_mul(np, Fcb) - 2 * fx_mul(nq, Fpb));
    // the frame's rotation (norms do not change under it)
    Wk += fx_msub(npb, nq, nqb, np);
    Wp += fx_msub(nqb, kn, knb, nq);
    Wq += fx_msub(knb, np, npb, kn);
    // (kn, np, nq) = (kr, pr, qr) / |n'|
    t = fx_prod<3>(knb, kn);
    fx_mac(t, npb, np);
    fx_mac(t, nqb, nq);
    const fxs dot = fx_split(fx_val(t));
    auto norm = [&](fxs xb, fxs x) {
      const fx r = (((fx)xb.h << 30) + xb.l) - fx_mul(x, dot);
      return fx_split(fx_mul(fx_split(r), inv));
    };
    const fxs krb = norm(knb, kn), prb = norm(npb, np), qrb = norm(nqb, nq);
    const volatile fx* pl = l < 2 ? pc + kFxL * l : pc + kFxProj3;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (m >= 2 && !helio) break;
      t = fx_prod<3>(krb, fx_unpack(pl[m]));
      fx_mac(t, prb, fx_unpack(pl[kFxV + m]));
      fx_mac(t, qrb, fx_unpack(pl[2 * kFxV + m]));
      obb[m] += fx_val(t);
    }
  }
  // the links' angles carry f k.delta_t / 2: (a / 3) (th_{l+1} - th_{l+2}) on k.n'_l (angles by link)
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    const int tl = kFtL + kFtLink * l;
    const fx d = l == 0 ? th1 - th2 : (l == 1 ? th2 - th0 : th0 - th1);
    const fxs kb = fx_split(fx_mul(fx_split(d), a3s));
    Wq += fx_mul(kb, fx_split(tape.ld(tl + kFtP)));
    Wp -= fx_mul(kb, fx_split(tape.ld(tl + kFtQ)));
    const volatile fx* pl = l < 2 ? pc + kFxL * l : pc + kFxProj3;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (m >= 2 && !helio) break;
      obb[m] += fx_mul(kb, fx_unpack(pl[m]));
    }
  }
  // orbit basis b = (cos 2 alpha, sin 2 alpha, cos alpha, sin alpha) or (cos phi_0, sin phi_0)
  const int e0 = E + Es - 2097, e = min(e0, kFxMostExpo), es = min(Es - 1078, kFxMostExpo);
  if (helio) {
    const fxs c = fx_split(tape.ld(kFtC)), s = fx_split(tape.ld(kFtS));
    fxa q = fx_sq0<1>();
    fx_macsq(q, s);
    const fxs c2 = fx_split(kFxOne - 2 * fx_valsq(q)), s2 = fx_split(2 * fx_mul(s, c));
    const fx r2 = fx_msub(c2, fx_split(obb[1]), s2, fx_split(obb[0]));
    const fx r1 = fx_msub(c, fx_split(obb[3]), s, fx_split(obb[2]));
    o.alpha = fx_to_double(2 * r2 + r1, e);
    o.geo = 0.0;
  } else {
    const fxs gc = fx_split(tape.ld(kFtGc)), gs = fx_split(tape.ld(kFtGs));
    o.alpha = 0.0;
    o.geo = fx_to_double(fx_msub(gc, fx_split(obb[1]), gs, fx_split(obb[0])), e);
  }
  o.th = fx_to_double(th0 + th1 + th2, e);
  o.lnA = fx_to_double(lnA, e);
  o.W[0] = fx_to_double(Wk, e);
  o.W[1] = fx_to_double(Wp, e);
  o.W[2] = fx_to_double(Wq, e);
  if (!some) o.th = o.lnA = o.alpha = o.geo = o.W[0] = o.W[1] = o.W[2] = 0.0;   // not the sums' rounding
  o.Ap = make_double2(fx_to_double(Apb[0], es), 0.0);
  o.Ac = make_double2(fx_to_double(Acb[0], es), 0.0);
  if (pair) {
    o.Ap.y = fx_to_double(Apb[1], es);
    o.Ac.y = fx_to_double(Acb[1], es);
  }
  if (max(e0, Es - 1078) > kFxMostExpo) {   // where floating point may overflow
    const double p = __hiloint2double(min(e0 - e + 1023, 0x7ff) << 20, 0), pa = __hiloint2double((Es - 1078 - es + 1023) << 20, 0);
    o.th *= p;
    o.lnA *= p;
    o.alpha *= p;
    o.geo *= p;
    for (int i = 0; i < 3; ++i) o.W[i] *= p;
    o.Ap = make_double2(o.Ap.x * pa, o.Ap.y * pa);
    o.Ac = make_double2(o.Ac.x * pa, o.Ac.y * pa);
  }
}

// Sums of one bin's sweeps over its modes; the factors common to the modes are applied once per bin (fx_bin_grad): ln amplitude; v d/dv of
// the phase and t_f chains; q, iota, phi_c, t_c; psib v^-2 - 2 Db v^-2 and psib v^-1 - Db v^-1 (chi1, chi2 enter P3 and P4
// alone); rotation; Doppler, f R-weighted cos and sin; Mtot through the taper and the paired mode.
enum : int { kGlnA, kGvM, kGq, kGio, kGph, kGtc, kGx3, kGx4, kGW, kGdc = kGW + 3, kGds, kGMx, kGSums };
struct FxBinAcc {       // in registers
  double v[kGSums];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < kGSums; ++i) v[i] = 0.0;
  }
  __device__ __forceinline__ double get(int i) const { return v[i]; }
  __device__ __forceinline__ void add(int i, double x) { v[i] += x; }
  __device__ __forceinline__ void mac(int i, double x, double y) { v[i] = fma(x, y, v[i]); }
};
template <int STRIDE>
struct FxBinAccShared {   // in a thread's column of shared memory: 28 registers less across the sweep
  volatile double* v;
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < kGSums; ++i) v[i * STRIDE] = 0.0;
  }
  __device__ __forceinline__ double get(int i) const { return v[i * STRIDE]; }
  __device__ __forceinline__ void add(int i, double x) { v[i * STRIDE] = v[i * STRIDE] + x; }
  __device__ __forceinline__ void mac(int i, double x, double y) { v[i * STRIDE] = fma(x, y, v[i * STRIDE]); }
};
// Reverse sweep of one unit, added to the bin's sums; the PN chain in FP64. fm13 = f^(-1/3), invf = 1/f, fR = 2 pi f R, n2pif = -2 pi f. (t_f's part of the
// chain in double words saved 14 FP64 FMAs a unit and no time: the kernel waits on dependent operations.)
template <int SST, class Tape, class BinAcc>
__device__ __forceinline__ void mode_bwd_fx(const DetDev& D, const SampleCoef& S, const SampleGrad& SG, int md, int md2, const FxBin& B,
                                            double fm13, double invf, double fR, double n2pif, fx a3, const volatile fx* seeds, int Es, BinAcc& g,
                                            const fx* __restrict__ pc, const Tape& tape) {
  const ModeCoef& C = S.md[md];
  const ModeGrad& CG = SG.md[md];
  const double v = C.cm * B.f13;
  const double w = __longlong_as_double(tape.ld(kFtW)), amp = __longlong_as_double(tape.ld(kFtAmp0)) * w;
  if (fx_expo(amp) == 0) return;
  double2 Ap, Ac;
  if constexpr (Tape::kChain) {
    Ap = make_double2(__longlong_as_double(tape.ld(kFtWeights)), __longlong_as_double(tape.ld(kFtWeights + 1)));
    Ac = make_double2(__longlong_as_double(tape.ld(kFtWeights + 2)), __longlong_as_double(tape.ld(kFtWeights + 3)));
  } else {
    fx_weights(S, C, md2 >= 0 ? &S.md[md2] : nullptr, amp, v, Ap, Ac);
  }
  FxBwd o;
  fx_bwd<SST>(B, a3, seeds, Es, Ap, Ac, md2 >= 0, D.orbit == 0, pc, tape, o);
  FxChain h;
  if constexpr (Tape::kChain) {
    auto ld = [&](int i) { return __longlong_as_double(tape.ld(kFtChain + i)); };
    h = FxChain{ld(0), ld(1), ld(2), ld(3), ld(4), ld(5), ld(6), ld(7)};
  } else {
    h = fx_chain(D, S, SG, C, CG, B, fm13, v, w, tape.ld(kFtC), tape.ld(kFtS));
  }
  // phase: ph0 = m phi_c / 2 pi + ..., -f t_c, -(m / 4 pi) Psi, -f k.x_c (turns)
  const double mh = md == 1 ? -0.5 : (md == 2 ? -1.5 : (md == 4 ? -2.0 : -1.0));   // -m/2
  const double psib = mh * o.th;                 // - mfac 2 pi th
  g.mac(kGph, -2.0, psib);
  // centre's Doppler term -f k.x_c, x_c = R (cos alpha, sin alpha, 0)
  const double fth = -fR * o.th, fc = fth * h.co, fs = fth * h.so;
  g.add(kGdc, fc);
  g.add(kGds, fs);
#pragma unroll
  for (int i = 0; i < 3; ++i) g.add(kGW + i, o.W[i]);
  const double alphab = fma(S.k[1], fc, fma(-S.k[0], fs, o.alpha));
  double tfb = alphab * D.rate_rad;
  if (D.orbit != 0) tfb = fma(o.geo, D.geo_rate_rad, tfb);
  g.add(kGtc, fma(n2pif, o.th, tfb));   // frac(f t_c); t_f = t_c + (m/(12 pi f)) D(v)
  const double Db = tfb * (C.tffac * invf);
  // amplitude ~ M^(5/6) ... f^(-7/6 + p/3) cm^p: dlnA_dM without the mode's own v is common to the modes
  g.add(kGlnA, o.lnA);
  g.mac(kGMx, o.lnA, h.tap);
  double vM = fma(psib, h.dv, Db * h.ddv);
  if (C.p != 0) vM += C.p == 1 ? o.lnA : 2.0 * o.lnA;
  double q = fma(psib, h.pq, fma(Db, h.dq, o.lnA * CG.dlnA_dq));
  g.mac(kGx4, h.iv, psib - Db);
  g.mac(kGx3, h.iv * h.iv, fma(-2.0, Db, psib));
  // polarisation weights: Ac carries 2 Pc
  double io = amp * fma(o.Ap.x, CG.dPp_di, o.Ac.x * (2.0 * CG.dPc_di));
  if (md2 >= 0) {
    const double2 apb = make_double2(amp * o.Ap.x, amp * o.Ap.y), acb = make_double2(amp * o.Ac.x, amp * o.Ac.y);
    const ModeGrad& CG2 = SG.md[md2];
    const double2 kap = make_double2(S.k32.x * (v * v), S.k32.y * (v * v));
    const double Pp2 = S.md[md2].Pp, Pc22 = S.md[md2].Pc2;
    io += (apb.x * kap.x + apb.y * kap.y) * CG2.dPp_di + 2.0 * (acb.x * kap.x + acb.y * kap.y) * CG2.dPc_di;
    const double2 kb = make_double2(apb.x * Pp2 + acb.x * Pc22, apb.y * Pp2 + acb.y * Pc22);   // kappa-bar
    // kappa = k32 v^2; only ln(amp2 / amp1) varies with theta (M, q), see mode_bwd
    const double lnrb = v * v * (kb.x * S.k32.x + kb.y * S.k32.y);
    g.mac(kGMx, lnrb, CG2.dlnA_dM - CG.dlnA_dM);
    q = fma(lnrb, CG2.dlnA_dq - CG.dlnA_dq, q);
    vM = fma(2.0, lnrb, vM);
  }
  g.add(kGvM, vM);
  g.add(kGq, q);
  g.add(kGio, io);
}

// The bin's theta components from its sums, with the rotation cotangents in g.k. th: the sample's parameters enter through
// SampleGrad alone: d ln v / d Mtot = 1 / (3 Mtot) = dcm_dM / cm.
template <class BinAcc>
__device__ __forceinline__ void fx_bin_grad(const SampleCoef& S, const SampleGrad& SG, const BinAcc& a, GradAcc& g) {
  const double m3 = SG.md[0].dcm_dM / S.md[0].cm;    // 1 / (3 Mtot)
  const double lnA = a.get(kGlnA), x3 = a.get(kGx3), x4 = a.get(kGx4), dc = a.get(kGdc), ds = a.get(kGds);
  g.M = fma(a.get(kGvM), m3, fma(lnA, 2.5 * m3, a.get(kGMx)));   // dlnA_dM = 5 / (6 Mtot)
  g.q = a.get(kGq);
  g.c1 = fma(SG.dP3_dc1, x3, SG.dP4_dc1 * x4);
  g.c2 = fma(SG.dP3_dc2, x3, SG.dP4_dc2 * x4);
  g.dL = lnA * SG.dlnA_ddL;
  g.io = a.get(kGio);
  g.ph = a.get(kGph);
  g.tc = a.get(kGtc);
  g.k[0] = a.get(kGW);
  g.k[1] = a.get(kGW + 1) - fma(S.q[0], dc, S.q[1] * ds);
  g.k[2] = a.get(kGW + 2) + fma(S.p[0], dc, S.p[1] * ds);
}

// Component c of the frame vectors' cotangents (vec 0 k, 1 p, 2 q) that stand for the rotation cotangents W: with
// dk = w x k = w_q p - w_p q and dp . q = w_k, kbar = W_q p - W_p q and pbar = W_k q give W.w for every rotation w.
__device__ __forceinline__ double rotation_to_frame(const SampleCoef& S, const double W[3], int vec, int c) {
  return vec == 0 ? W[2] * S.p[c] - W[1] * S.q[c] : (vec == 1 ? W[0] * S.q[c] : 0.0);
}

// The bin's link seeds as integers: exponent Es of the largest (0: all vanish, and so does the bin's gradient), n = value 2^(1078 - Es) below 1/16.
template <int SST>
__device__ __forceinline__ int fx_seeds(const double2 pq[6], volatile fx* seeds) {
  int Es = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) Es = max(Es, max(fx_expo(pq[i].x), fx_expo(pq[i].y)));
  const int sh = 1078 - Es;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    seeds[2 * i * SST] = fx_from_bits(pq[i].x, sh);
    seeds[(2 * i + 1) * SST] = fx_from_bits(pq[i].y, sh);
  }
  return Es;
}

}  // namespace pe
