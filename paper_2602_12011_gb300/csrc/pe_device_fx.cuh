// pe_device_fx.cuh -- the FP64 path's (sample, mode, bin) unit with its response geometry in 64-bit
// fixed point (pe_fx.cuh): the same definitions as mode_bin (pe_device.cuh; arXiv:2602.12011 Sec. 2.1,
// Eq. eq_tf, eq_fd_resp, FD TDI).
//
// On the FP64 pipe stay the TaylorF2 phase, t_f far from t_c, the amplitudes and the PSD-weighted
// sums, which need FP64's range: about 35 of the 243 FP64 instructions that mode_bin issues per unit. The orbit's sine and cosine, the link vectors' projections and norms, the
// polarisation factors, the third-spacecraft and Doppler phases, the sincs and the TDI sums are Q60
// integers or, where only a correction below 2^-8 is formed, double words. Their errors are those
// of 2^-58 to 2^-56 of unit-sized quantities (root mean square), against 2^-54.5 for the FP64 ones.
//
// Amplitudes span many orders of magnitude along a grid, so a bin's sums are block floating point:
// the accumulators share one binary exponent per bin, taken from the largest amplitude so far, and
// the mode sum's smaller modes lose only bits below 2^-60 of it.
//
// Bound by the latency of dependent integer and double-word operations, at 62 % of the issue slots and 61 % of the FP64 pipe, so
// warps count: 1024 LISA samples of 2^22 s (five modes) take 24.3 ms in FP64, 5.75 ms here with 6 CTAs of 128 per SM and one sinc
// per call, 5.52 with pairs of them and the finer table, 4.95 with 8 CTAs (64 registers; 5.33 with 7, 5.37 with 9). The PN
// series as fixed-point Horner chains took 9 more FP64 operations off each unit and made it 6.2 ms.
#pragma once
#include "pe_device.cuh"
#include "pe_fx.cuh"

namespace pe {

// A detector takes this path where the formats' bounds hold (fill_fx, pe_api.cu): a = pi f L < 4 on its whole
// grid, an eccentricity below 0.05 (link lengths near the nominal arm), and indices below 2^31.

// (k c) 2^60 for the detector constant c = C 2^-(60 + sh): see DetDev::fx_*.
__device__ __forceinline__ fx fx_times_k(unsigned k, const FxConst& c) {
  const fxu lo = (fxu)k * (unsigned)c.C;
  const fxu hi = (fxu)k * (unsigned)(c.C >> 32) + (lo >> 32);   // k C = hi 2^32 + low word of lo
  return c.sh >= 32 ? (fx)(hi >> (c.sh - 32)) : (fx)((hi << (32 - c.sh)) | ((unsigned)lo >> c.sh));
}

// What the units of one (detector, sample) pair share, in shared memory (kFxProj words, 16-byte aligned): for the links l = 0, 1
// proj_coef's forms over the nominal arm at kFxL l + kFxV v + m, m < 4 split for multiplication (h in the high word, l in the
// low one; read two at a time) and the constant m = 4 a plain Q60; k_x, k_y (split); the centre's angle at t_c (turns);
// per mode m / (12 pi) cm^-5 as a double word, and the amplitude times the polarisation weights (doubles).
// Entries kFxProj3 + kFxV v + m (m < 4): the third link's forms, minus the others' sum (fx_proj3; the reverse sweep's).
constexpr int kFxV = 6, kFxL = 3 * kFxV;
enum : int { kFpK = 2 * kFxL, kFpAlpha = kFpK + 2, kFpTau, kFpPp = kFpTau + kNModes, kFpPc = kFpPp + kNModes,
             kFpEnd = kFpPc + kNModes };
constexpr int kFxProj = ((kFpEnd > kProj ? kFpEnd : kProj) + 1) / 2 * 2;   // kernels of both units share the array
constexpr int kFxProj3 = kFxProj, kFxProjAll = kFxProj + kFxL;
__device__ __forceinline__ fx fx_pack(fxs s) { return ((fx)s.h << 32) | (unsigned)s.l; }
__device__ __forceinline__ fxs fx_unpack(fx p) {
  fxs r;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(r.l), "=r"(r.h) : "l"(p));
  return r;
}
// Two packed words at p (16-byte aligned, shared memory); volatile, so that no form stays in registers across the links
__device__ __forceinline__ void fx_ld2(const volatile fx* p, fxs& a, fxs& b) {
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(a.l), "=r"(a.h), "=r"(b.l), "=r"(b.h)
               : "r"((unsigned)__cvta_generic_to_shared(const_cast<const fx*>(p))));
}
__device__ __forceinline__ void fx_proj_prologue(const DetDev& D, const SampleCoef& S, fx* pc) {
  __syncthreads();
  for (int i = threadIdx.x; i < 30 + kFpEnd - kFpK; i += blockDim.x) {
    if (i < 30) {   // proj_coef's order: 15 l + 5 v + m
      const fx q = fx_from_bits(proj_coef(D, S, i) * D.fx_iL, 60);
      pc[i / 5 * kFxV + i % 5] = i % 5 == 4 ? q : fx_pack(fx_split(q));
      continue;
    }
    const int j = i - 30 + kFpK;
    fx q = 0;
    if (j < kFpAlpha) {
      q = fx_pack(fx_split(fx_from_bits(S.k[j - kFpK], 60)));
    } else if (j == kFpAlpha) {
      q = (fx)fx_turns(fma(S.tc, D.rate_t, D.alpha0_t));
    } else if (j < kFpPp) {
      const ModeCoef& C = S.md[j - kFpTau];
      const float2 w = to_dw(C.tffac * C.icm5);
      q = ((fx)__float_as_int(w.y) << 32) | (unsigned)__float_as_int(w.x);
    } else {
      const ModeCoef& C = S.md[(j - kFpPp) % kNModes];
      q = __double_as_longlong(C.ampp * (j < kFpPc ? C.Pp : C.Pc2));
    }
    pc[j] = q;
  }
  __syncthreads();
}
__device__ __forceinline__ void fx_proj3(fx* pc) {   // after fx_proj_prologue; a barrier at the end
  const int i = threadIdx.x;
  if (i < kFxL && i % kFxV < 4) {
    const fxs a = fx_unpack(pc[i]), b = fx_unpack(pc[kFxL + i]);
    pc[kFxProj3 + i] = fx_pack(fx_split(-((((fx)a.h + b.h) << 30) + a.l + b.l)));
  }
  __syncthreads();
}
// p[0..3] . b + p[4] (geocentric: b has two entries and the constant is zero)
__device__ __forceinline__ fx fx_dot(const volatile fx* p, const fxs b[4], bool helio) {
  fxs c0, c1;
  fx_ld2(p, c0, c1);
  fxa s = fx_prod<2>(c0, b[0]);
  fx_mac(s, c1, b[1]);
  if (helio) {
    fx_ld2(p + 2, c0, c1);
    s.c += 2 * kFxLL;
    fx_mac(s, c0, b[2]);
    fx_mac(s, c1, b[3]);
    s.h += p[4];
  }
  return fx_val(s);
}

// Per-bin inputs shared by the modes of one bin.
struct FxBin {
  double f, f13, lnf3;
  fxu frc;             // f t_c modulo one turn
  fx a4;               // a / 4, a = pi f L
  fxs at3, fR;         // f L / 6; f R 2^-fx_rsh
  int b;
};
__device__ __forceinline__ void load_bin_fx(const DetDev& D, int b, double tc, FxBin& B) {
  B.f = D.f[b];
  B.f13 = D.f13[b];
  B.lnf3 = D.lnf3[b];
  B.frc = fx_cycles(B.f, tc);
  const unsigned k = (unsigned)(D.k0 + b);
  B.a4 = fx_times_k(k, D.fx_a4);
  B.at3 = fx_split(fx_times_k(k, D.fx_at3));
  B.fR = fx_split(fx_times_k(k, D.fx_fR));
  B.b = b;
}

// Mode-summed link products of one bin (see XYZAcc), in units of 2^(E - 1079): E is the largest
// biased exponent of an amplitude so far (0: none yet). The twelve sums (S_r, S_i, M_r, M_i of link l at 4 l)
// stay in the thread's column of shared memory, which frees 24 registers and lets the link loop stay
// rolled.
constexpr int kFxSums = 12;
template <int STRIDE>
struct FxAccT {
  static constexpr int kStride = STRIDE;
  volatile fx* s;      // entry i at s[i * kStride]
  int E;
};
using FxAcc = FxAccT<kTileBins>;
template <class Acc>
__device__ __forceinline__ void fx_zero(Acc& a, fx* col) {
  a.s = col;
#pragma unroll
  for (int i = 0; i < kFxSums; ++i) a.s[i * Acc::kStride] = 0;
  a.E = 0;
}
constexpr int kFxLeastE = 64;   // amplitudes below 2^-959 count as 0: above, a zero beside them converts to 0 (fx_from_bits)
constexpr float kFxTauMax = 8192.f;
__device__ __forceinline__ int fx_expo(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// The orbit's basis from the centre's angle (heliocentric: cos 2 alpha, sin 2 alpha, cos alpha, sin alpha) or the
// constellation's (geocentric: its cosine and sine).
__device__ __forceinline__ void fx_basis(fxc g, bool helio, fxs ob[4]) {
  const fxs cs = fx_split(g.c), ss = fx_split(g.s);
  if (helio) {
    fxa q = fx_sq0<1>();
    fx_macsq(q, ss);
    ob[0] = fx_split(kFxOne - 2 * fx_valsq(q));   // cos 2 alpha = 1 - 2 sin^2 alpha
    ob[1] = fx_split(2 * fx_mul(ss, cs));
    ob[2] = cs;
    ob[3] = ss;
  } else {
    ob[0] = cs;
    ob[1] = ss;
    ob[2] = ob[3] = fxs{0, 0};
  }
}

// Fields of a unit's tape for the reverse sweep (pe_adjoint_fx.cuh): the centre's and the constellation's cosine and sine,
// the amplitude before the taper and the taper's weight (doubles' bits), and per link l the projections of the link
// vector over the arm, its inverse length, the factor e^{i phase}, sinc(a (1 +- k.n)) and their derivatives in u.
enum : int { kFtC = 0, kFtS = 1, kFtGc = 2, kFtGs = 3, kFtAmp0 = 4, kFtW = 5, kFtL = 6, kFtLink = 10, kFtFields = 36 };
enum : int { kFtK = 0, kFtP = 1, kFtQ = 2, kFtInv = 3, kFtEc = 4, kFtEs = 5, kFtSp = 6, kFtSm = 7, kFtDp = 8, kFtDm = 9 };
struct FxNoTape {
  static constexpr bool kOn = false;
  __device__ __forceinline__ void st(int, fx) const {}
};

// One unit's link products, added to the bin's sums: phu the mode's phase (turns), Apx, Acx the polarisation weights
// times the amplitude; for a paired second mode Ap (its imaginary part read) and Acyd complete them, scaled by
// 2^ash.
template <class Acc, class Tape = FxNoTape>
__device__ __forceinline__ void fx_links(fxs at3, fx a4, fxu phu, fxs Apx, fxs Acx, const double2* Ap, double Acyd, int ash,
                                         const fxs ob[4], bool helio, Acc& acc, const FxCis* __restrict__ tab,
                                         const FxSinc* __restrict__ stab, const fx* __restrict__ pc, Tape tape = Tape()) {
  const fxs a4s = fx_split(a4);
  // --- links (row A5): projections of the link vectors over the nominal arm; the three sum to zero.
  // Third-spacecraft phases f k.delta_t / 2 in turns: delta_0 - delta_1, delta_1 - delta_2 and
  // delta_2 - delta_0 are the link vectors and the offsets sum to zero, so delta_0 = (n_0 - n_2)/3,
  // delta_1 = (n_1 - n_0)/3 and delta_2 is minus both
  const fx kn0 = fx_dot(pc, ob, helio), kn1 = fx_dot(pc + kFxL, ob, helio), kn2 = -(kn0 + kn1);
  const fxu e0 = (fxu)fx_mul(fx_split(kn0 - kn2), at3) << 4;
  const fxu e1 = (fxu)fx_mul(fx_split(kn1 - kn0), at3) << 4;
  fx np = 0, nq = 0;   // minus the sums of the earlier links' projections
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    fx pr = np, qr = nq;
    if (l < 2) {
      pr = fx_dot(pc + kFxL * l + kFxV, ob, helio);
      qr = fx_dot(pc + kFxL * l + 2 * kFxV, ob, helio);
      np -= pr;
      nq -= qr;
    }
    const fxs k0 = fx_split(l == 0 ? kn0 : (l == 1 ? kn1 : kn2)), p0 = fx_split(pr), q0 = fx_split(qr);
    fxa n2 = fx_sq0<3>();
    fx_macsq(n2, k0);
    fx_macsq(n2, p0);
    fx_macsq(n2, q0);
    const fx invq = fx_rsqrt(fx_valsq(n2));
    const fxs inv = fx_split(invq);
    const fx w4 = fx_mul(fx_split(fx_mul(k0, inv)), a4s);
    const fx p1 = fx_mul(p0, inv), q1 = fx_mul(q0, inv);
    // F+ = (n.p)^2 - (n.q)^2, Fx / 2 = (n.p)(n.q) (the 2 is in Ac)
    const fxs Fp = fx_split(fx_mul(fx_split(p1 - q1), fx_split(p1 + q1)));
    const fxs Fc = fx_split(fx_mul(fx_split(p1), fx_split(q1)));
    fxs gx, gy;
    if (Ap) {
      const fxs Apy = fx_split(fx_from_bits(Ap->y, ash)), Acy = fx_split(fx_from_bits(Acyd, ash));
      gx = fx_split(fx_msub(Apx, Fp, Acy, Fc));
      fxa g = fx_prod<2>(Apy, Fp);
      fx_mac(g, Acx, Fc);
      gy = fx_split(fx_val(g));
    } else {
      gx = fx_split(fx_mul(Apx, Fp));
      gy = fx_split(fx_mul(Acx, Fc));
    }
    // the third spacecraft is 2, 0, 1 for l = 0, 1, 2
    const fxc e = fx_cis(l == 0 ? phu - (e0 + e1) : phu + (l == 1 ? e0 : e1), tab);
    const fxs ec = fx_split(e.c), es = fx_split(e.s);
    const int tl = kFtL + kFtLink * l;
    if constexpr (Tape::kOn) {
      tape.st(tl + kFtK, l == 0 ? kn0 : (l == 1 ? kn1 : kn2));
      tape.st(tl + kFtP, pr);
      tape.st(tl + kFtQ, qr);
      tape.st(tl + kFtInv, invq);
      tape.st(tl + kFtEc, e.c);
      tape.st(tl + kFtEs, e.s);
    }
    const fxs Gr = fx_split(fx_msub(gx, ec, gy, es));
    fxa gi = fx_prod<2>(gx, es);
    fx_mac(gi, gy, ec);
    const fxs Gi = fx_split(fx_val(gi));
    // --- sinc(a (1 +- k.n)) and the link's products for the TDI brackets (row A6; see XYZAcc)
    volatile fx* as = acc.s + 4 * l * Acc::kStride;
    const fx2 sv = fx_sinc2(a4 + w4, a4 - w4, stab);
    const fxs sp = fx_split(sv.p), sm = fx_split(sv.m);
    if constexpr (Tape::kOn) {
      const fx2 dv = fx_sinc2(a4 + w4, a4 - w4, stab + kFxSincTab);   // the derivative's table follows
      tape.st(tl + kFtSp, sv.p);
      tape.st(tl + kFtSm, sv.m);
      tape.st(tl + kFtDp, dv.p);
      tape.st(tl + kFtDm, dv.m);
    }
    as[0] = as[0] + fx_mul(Gr, sp);
    as[Acc::kStride] = as[Acc::kStride] + fx_mul(Gi, sp);
    as[2 * Acc::kStride] = as[2 * Acc::kStride] + fx_mul(Gr, sm);
    as[3 * Acc::kStride] = as[3 * Acc::kStride] + fx_mul(Gi, sm);
  }
}

template <class Acc, class Tape = FxNoTape>
__device__ __forceinline__ void mode_bin_fx(const DetDev& D, const SampleCoef& S, const ModeCoef& C, const FxBin& B,
                                            Acc& acc, const FxCis* __restrict__ tab, const FxSinc* __restrict__ stab,
                                            const fx* __restrict__ pc, int md, const ModeCoef* C2 = nullptr,
                                            Tape tape = Tape()) {
  // --- waveform and time-frequency map (rows A2, A3), as mode_bin
  const double v = C.cm * B.f13;
  const double lnv = C.lncm + B.lnf3;
  const double iv5 = C.icm5 * D.fm53[B.b];
  double poly = S.P[7];
#pragma unroll
  for (int k = 6; k >= 0; --k) poly = fma(poly, v, S.P[k]);
  const double q56 = fma(S.Q6, v, S.Q5);
  const double psi_pn = fma(iv5, poly, lnv * q56);
  // t_f - t_c = (m / 12 pi) f^-1 v dPsi/dv = (m / 12 pi) cm^-5 f^(-8/3) (sum_k Pd_k v^k + v^5 (Q5 + Q6 v (1 + ln v)))
  // in double words (2^-45): below kFxTauMax seconds from t_c the heliocentric angle it turns the orbit by
  // is then known to 2^-57 turn, and only farther out, and for a geocentric orbit, is t_f formed in FP64
  // (FP64 operations per unit 43 -> 35 over the prior)
  const df vw = dfl_mul(C.cmw, D.f13w[B.b]);
  df tau;
  {
    df dpol = S.Pdw[7];
#pragma unroll
    for (int k = 6; k >= 2; --k) dpol = dfl_add(dfl_mul(dpol, vw), S.Pdw[k]);
    const df v2 = dfl_mul(vw, vw);
    dpol = dfl_add(S.Pdw[0], dfl_mul(v2, dpol));                 // Pd_1 = 0
    const df q6v = dfl_mul(S.Q6w, vw);
    const df q = dfl_add(S.Q5w, dfl_add(q6v, dfl_mul(q6v, df_from_bits(lnv))));
    dpol = dfl_add(dpol, dfl_mul(dfl_mul(dfl_mul(v2, v2), vw), q));
    const fx kw = pc[kFpTau + md];
    tau = dfl_mul(dfl_mul(df_make(__int_as_float((int)kw), __int_as_float((int)(kw >> 32))), D.fm83w[B.b]), dpol);
  }
  const bool helio = D.orbit == 0;
  fxu alpha;           // the centre's angle and, for a geocentric orbit, the constellation's
  fxu geo = 0;
  if (helio && fabsf(tau.x) < kFxTauMax) {
    // the series' terms may cancel and leave a low word beyond fx_from_dw's bound: normalised first
    const df a = dfl_mul(tau, D.ratew);
    alpha = (fxu)pc[kFpAlpha] + ((fxu)fx_from_dw(two_sum(a.x, a.y)) << 4);
  } else {
    double dpol = S.Pd[7];
#pragma unroll 1
    for (int k = 6; k >= 0; --k) dpol = fma(dpol, v, S.Pd[k]);
    const double fm13 = D.fm13[B.b];
    const double dv = fma(iv5, dpol, fma(S.Q6 * v, lnv, q56));
    const double tf = fma(C.tffac * (fm13 * fm13 * fm13), dv, S.tc);
    alpha = fx_turns(fma(tf, D.rate_t, D.alpha0_t));
    geo = fx_turns(tf * D.geo_rate_t);
  }
  // polarisation weights times the amplitude (complex for a paired second mode), as integers below
  // 1/8 in units of 2^(E - 1079)
  const double fp = C.p == 0 ? D.fm76[B.b] : (C.p == 1 ? D.fm56[B.b] : D.fm12[B.b]);
  double2 Ap, Ac;
  double w = 1.0;
  if (C2) {
    const double v2 = v * v, amp = C.ampp * fp;
    const double kr = S.k32.x * v2, ki = S.k32.y * v2;
    Ap = make_double2(amp * fma(kr, C2->Pp, C.Pp), amp * (ki * C2->Pp));
    Ac = make_double2(amp * fma(kr, C2->Pc2, C.Pc2), amp * (ki * C2->Pc2));
  } else {
    Ap = make_double2(fp * __longlong_as_double(pc[kFpPp + md]), 0.0);
    Ac = make_double2(fp * __longlong_as_double(pc[kFpPc + md]), 0.0);
  }
  if (dlt_pos(C.ftap, B.f)) {
    const double span = C.fend - C.ftap;
    const double zt = span / (C.fend - B.f) - span / (B.f - C.ftap);
    w = (zt > 700.0) ? 0.0 : 1.0 / (1.0 + exp(zt));
    Ap = make_double2(Ap.x * w, Ap.y * w);
    Ac = make_double2(Ac.x * w, Ac.y * w);
  }
  if constexpr (Tape::kOn) {
    tape.st(kFtAmp0, __double_as_longlong(C.ampp * fp));
    tape.st(kFtW, __double_as_longlong(w));
  }
  int E = max(fx_expo(Ap.x), fx_expo(Ac.x));
  if (C2) E = max(E, max(fx_expo(Ap.y), fx_expo(Ac.y)));
  // below kFxLeastE the weights vanish (the unit adds nothing; its tape still serves the weights' own derivatives)
  if (!Tape::kOn && E < kFxLeastE) return;
  if (E > acc.E) {
    if (acc.E > 0) {
      const int sh = min(62, E - acc.E);
#pragma unroll 1
      for (int i = 0; i < kFxSums; ++i) acc.s[i * Acc::kStride] = (acc.s[i * Acc::kStride] + (1LL << (sh - 1))) >> sh;
    }
    acc.E = E;
  }
  const int ash = 1079 - acc.E;
  const bool some = E >= kFxLeastE;
  const fxs Apx = some ? fx_split(fx_from_bits(Ap.x, ash)) : fxs{0, 0}, Acx = some ? fx_split(fx_from_bits(Ac.x, ash)) : fxs{0, 0};
  // --- orbit at t_f (row A4): mode phase in turns, the centre's Doppler term f k.x_c = f R (k_x cos + k_y sin)
  // included, and the offsets' basis
  const fxc ca = fx_cis(alpha, tab);
  fxs kx, ky;
  fx_ld2(pc + kFpK, kx, ky);
  fxa kc = fx_prod<2>(kx, fx_split(ca.c));
  fx_mac(kc, ky, fx_split(ca.s));
  const fxu phu = fx_turns(fma(-C.mfac, psi_pn, C.ph0)) - B.frc -
                  ((fxu)fx_mul(fx_split(fx_val(kc)), B.fR) << (4 + D.fx_rsh));
  fxs ob[4];
  const fxc cg = helio ? ca : fx_cis(geo, tab);
  fx_basis(cg, helio, ob);
  if constexpr (Tape::kOn) {
    tape.st(kFtC, ca.c);
    tape.st(kFtS, ca.s);
    if (!helio) {
      tape.st(kFtGc, cg.c);
      tape.st(kFtGs, cg.s);
    }
  }
  fx_links(B.at3, B.a4, phu, Apx, Acx, C2 && some ? &Ap : nullptr, Ac.y, ash, ob, helio, acc, tab, stab, pc, tape);
}

// n 2^e as a double, the power of two added to the exponent field (0 where the result would lie below 2^-1020); e <= kFxMostExpo
constexpr int kFxMostExpo = 960;   // n's largest power of two then still fits a double
__device__ __forceinline__ double fx_to_double(fx n, int e) {
  const double d = __ll2double_rn(n);
  const int hi = __double2hiint(d);
  return fx_expo(d) + e > 2 ? __hiloint2double(hi + (e << 20), __double2loint(d)) : 0.0;
}

// Half the brackets X', Y', Z' of one bin's sums (xyz_final), and A/E/T from them (aet_from_xyz). Each unit's |G| is below
// 0.2 and a bin has four at most, so the brackets P and Q stay below 1.6, X', Y', Z' below 3.2 and
// the half sums of A/E/T below 6.4.
template <class Acc>
__device__ __forceinline__ void xyz_from_fx(const Acc& a, fxs zr, fxs zi, fx xr[3], fx xi[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const volatile fx* ac = a.s + 4 * c * Acc::kStride;                  // S_r, S_i, M_r, M_i of link c
    const volatile fx* al = a.s + 4 * ((c + 2) % 3) * Acc::kStride;      // and of link c + 2
    const fxs qr = fx_split(al[2 * Acc::kStride] - ac[0]), qi = fx_split(al[3 * Acc::kStride] - ac[Acc::kStride]);
    // halved: two more quarter units for the bit that drops
    xr[c] = ((al[0] - ac[2 * Acc::kStride]) + fx_msub<2>(zr, qr, zi, qi)) >> 1;
    fxa t = fx_prod<4>(zr, qi);
    fx_mac(t, zi, qr);
    xi[c] = ((al[Acc::kStride] - ac[3 * Acc::kStride]) + fx_val(t)) >> 1;
  }
}
template <class Acc>
__device__ __forceinline__ void aet_from_fx(const Acc& a, double2 z, double2 o[3]) {
  fx xr[3], xi[3];
  xyz_from_fx(a, fx_split(fx_from_bits(z.x, 60)), fx_split(fx_from_bits(z.y, 60)), xr, xi);
  // one unit of the halved sums is 2^e; amplitudes beyond 2^1015 (and infinite ones) count as 2^1015, whose <h|h> overflows too
  const int e = min(a.E - 1078, kFxMostExpo);
  o[0] = make_double2(fx_to_double(xr[2] - xr[0], e), fx_to_double(xi[2] - xi[0], e));
  o[1] = make_double2(fx_to_double(xr[0] - 2 * xr[1] + xr[2], e), fx_to_double(xi[0] - 2 * xi[1] + xi[2], e));
  o[2] = make_double2(fx_to_double(xr[0] + xr[1] + xr[2], e), fx_to_double(xi[0] + xi[1] + xi[2], e));
}

// Adds every active mode of one sample at one bin ((2,2) and (3,2) through one unit when both are
// active), then forms A/E/T. D0: the detector whose copy of the tables is read (the set's first, so that one copy
// stays in L1); col: the thread's column of kFxSums x kTileBins words of shared memory; expo (nullable): the sums' exponent (FxAccT).
__device__ __forceinline__ void bin_aet_fx(const DetDev& D, const SampleCoef& S, int b, double2 o[3],
                                           const DetDev& D0, const fx* __restrict__ pc, fx* col, int* expo = nullptr) {
  FxBin B;
  load_bin_fx(D, b, S.tc, B);
  FxAcc a;
  fx_zero(a, col);
#pragma unroll 1
  for (int md = 0; md < kNModes; ++md) {
    if (md == 3 && S.pair32) continue;
    const ModeCoef& C = S.md[md];
    if (!C.active || !dlt_pos(B.f, C.fend)) continue;
    mode_bin_fx(D, S, C, B, a, D0.fcis, D0.fsinc, pc, md, (md == 0 && S.pair32) ? &S.md[3] : nullptr);
  }
  aet_from_fx(a, D.z[b], o);
  if (expo) *expo = a.E;
}

}  // namespace pe
